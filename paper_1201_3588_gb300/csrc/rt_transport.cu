// rt_transport.cu -- photon-package transport kernels of librt_gb300.
//
// A package (Sec. 2) leaves the star with constant energy eps at a frequency bin
// drawn from the stellar spectrum, samples an optical depth tau = -ln(xi), and
// walks the grid of cubes and subcubes cell by cell, spending
// rho * kappa_ext * path of its tau in each cell. Where tau runs out it
// interacts: with probability kappa_sca / kappa_ext it scatters by the
// Henyey-Greenstein phase function, otherwise it is absorbed -- the cell's count
// of absorptions rises by one (an exact integer; eps is constant) and a package
// of the same energy leaves the absorption spot isotropically at a frequency
// drawn from the re-emission spectrum. A package that leaves the domain is binned
// into the escaped spectrum.
//
// Random numbers: Philox4x32-10 (Salmon et al. 2011), key = seed, counter =
// (package id lo, id hi, event index, block). Event 0 is the emission and uses
// one block: {bin, mu, phi, tau}. Interaction k uses block 0 = {albedo test,
// species, mu, phi} and block 1 = {tau, energy position, bin, -}. Each 32-bit word
// maps to the midpoint of one of 2^23 equal sub-intervals of (0,1).
//
// Re-emission bin: the three rules of Sec. 2 (the Bjorkman & Wood difference
// spectrum, its omission, a frozen temperature) are all mixtures over the
// temperature-table intervals: an energy per gram u is drawn uniformly in
// [u_lo, u_hi] (BW: [n, n+1] eps/M; no correction: [0, max(n eps/M, S(t_min))];
// frozen: [0, S(T_frozen)]), the table interval holding u is found in S(T), and
// the bin is drawn from that interval's normalised cumulative difference
// kappa_abs [P_b(T_{i+1}) - P_b(T_i)].
//
// Geometry: positions are in base-cube units. A point on a face belongs to the
// cell ahead of the direction of motion. After a face crossing the position is
// set exactly onto the face (exactly representable) and the other coordinates are
// clamped into the cell, so every crossing advances the cell index.

#include "rt_internal.h"

#include <math.h>

#include <type_traits>

namespace rt {
namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// ---------------------------------------------------------------- Philox
__device__ __forceinline__ uint4 philox10(uint4 c, uint2 k) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) {
      k.x += 0x9E3779B9u;
      k.y += 0xBB67AE85u;
    }
    unsigned hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
    unsigned hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
  }
  return c;
}

__device__ __forceinline__ uint4 draw(unsigned long long seed, unsigned long long id,
                                      unsigned event, unsigned block) {
  return philox10(make_uint4((unsigned)id, (unsigned)(id >> 32), event, block),
                  make_uint2((unsigned)seed, (unsigned)(seed >> 32)));
}

template <typename R>
__device__ __forceinline__ R unit(unsigned x) {
  return ((R)(x >> 9) + (R)0.5) * (R)(1.0 / 8388608.0);
}

// ---------------------------------------------------------------- math helpers
template <typename R> __device__ __forceinline__ R rsqrt_(R x);
template <> __device__ __forceinline__ float rsqrt_(float x) { return rsqrtf(x); }
template <> __device__ __forceinline__ double rsqrt_(double x) { return rsqrt(x); }

template <typename R>
__device__ __forceinline__ void sincos2pi(R xi, R* s, R* c);
template <> __device__ __forceinline__ void sincos2pi(float xi, float* s, float* c) {
  sincospif(2.0f * xi, s, c);
}
template <> __device__ __forceinline__ void sincos2pi(double xi, double* s, double* c) {
  sincospi(2.0 * xi, s, c);
}

template <typename R> __device__ __forceinline__ R log_(R x);
template <> __device__ __forceinline__ float log_(float x) { return logf(x); }
template <> __device__ __forceinline__ double log_(double x) { return log(x); }

// isotropic direction from two deviates
template <typename R>
__device__ __forceinline__ void isotropic(R xmu, R xphi, R d[3]) {
  R mu = (R)2 * xmu - (R)1;
  R s = sqrt(fmax((R)0, (R)1 - mu * mu));
  R sp, cp;
  sincos2pi(xphi, &sp, &cp);
  d[0] = s * cp;
  d[1] = s * sp;
  d[2] = mu;
}

// Henyey-Greenstein cos(theta) by inversion of its cumulative distribution
template <typename R>
__device__ __forceinline__ R hg_mu(R g, R xi) {
  if (fabs(g) < (R)1e-6) return (R)2 * xi - (R)1;
  R f = ((R)1 - g * g) / ((R)1 - g + (R)2 * g * xi);
  R mu = ((R)1 + g * g - f * f) / ((R)2 * g);
  return fmin((R)1, fmax((R)-1, mu));
}

// turn d by polar cosine mu and azimuth 2 pi xphi, azimuth counted from
// (dx dz, dy dz, -(1-dz^2))/sqrt(1-dz^2) towards (-dy, dx, 0)/sqrt(1-dz^2)
template <typename R>
__device__ __forceinline__ void turn(R d[3], R mu, R xphi) {
  R s = sqrt(fmax((R)0, (R)1 - mu * mu));
  R sp, cp;
  sincos2pi(xphi, &sp, &cp);
  R ux = d[0], uy = d[1], uz = d[2], nx, ny, nz;
  if (fabs(uz) > (R)0.99999) {
    nx = s * cp;
    ny = s * sp;
    nz = (uz > (R)0 ? mu : -mu);
  } else {
    R r2 = (R)1 - uz * uz;
    R ir = rsqrt_(r2);
    R r = r2 * ir;
    nx = mu * ux + s * (ux * uz * cp - uy * sp) * ir;
    ny = mu * uy + s * (uy * uz * cp + ux * sp) * ir;
    nz = mu * uz - s * r * cp;
  }
  R in = rsqrt_(nx * nx + ny * ny + nz * nz);
  d[0] = nx * in;
  d[1] = ny * in;
  d[2] = nz * in;
}

// first index whose normalised cumulative value exceeds xi (cdf[n-1] == 1)
__device__ __forceinline__ int search_cdf(const float* cdf, int n, float xi) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (cdf[mid] > xi) hi = mid; else lo = mid + 1;
  }
  return lo;
}

// ---------------------------------------------------------------- grid
template <typename R>
__device__ __forceinline__ int cell_index(R q, R d) {
  R f = floor(q);
  int i = (int)f;
  if (d < (R)0 && f == q) --i;
  return i;
}

// Leaf holding p when moving along d. Returns 0 inside, 1 outside, -1 malformed.
template <typename R>
__device__ __forceinline__ int locate(const DevGrid& g, const R p[3], const R d[3],
                                      int& leaf, int& level, int I[3]) {
  const int n = g.n_base;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    I[a] = cell_index(p[a], d[a]);
    if (I[a] < 0 || I[a] >= n) return 1;
  }
  int node = __ldg(&g.base[I[0] + n * (I[1] + n * I[2])]);
  int lev = 0;
  while (node < 0) {
    long long blk = -(long long)node - 1;
    if (blk >= g.n_blocks || lev >= g.max_level) return -1;
    ++lev;
    R sc = (R)(1 << lev);
    int oct = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      int j = cell_index(p[a] * sc, d[a]);
      int o = j - 2 * I[a];
      if ((unsigned)o > 1u) return -1;
      oct |= o << a;
      I[a] = j;
    }
    node = __ldg(&g.child[blk * 8 + oct]);
  }
  if ((long long)node >= g.n_leaves) return -1;
  leaf = node;
  level = lev;
  return 0;
}

// ---------------------------------------------------------------- package
template <typename R>
struct Pkg {
  R p[3], d[3];
  R inv[3];  // 1/d; +inf where d == 0 (of either sign)
  R tau;
  int bin;
  unsigned event;  // interactions so far
  unsigned long long id;
  unsigned dirs;  // the pool's walks: signs of the direction (see orient)
};

struct Tally {  // per-thread counters (plain kernel), flushed to the 64-bit device totals
  unsigned emitted, escaped, capped, absorptions, scatters, crossings, errors, clamped;
  unsigned levels;  // child-table reads of the walk
  unsigned peel_events, peel_crossings;  // peel-off sight lines and the cells they cross
};

// The pool counts crossings and tree reads per lane and everything rarer per warp in
// shared memory (nine counters in registers made the walks spill).
struct LaneTally {
  unsigned crossings, levels;
};

constexpr int kTallyWords = 16;  // per warp: kNumCounters words
static_assert(kNumCounters <= kTallyWords, "the counters fit a warp's words");

// a flush is forced once a counter passes 2^30: between two looks at them the pool adds at
// most 32 x 2^24 to a warp's and kWalkSteps x 2^24 to a lane's
constexpr unsigned kTallyFlushAt = 1u << 30;

// Cells a lane crosses at most before the warp looks whether lanes are idle: looking costs
// every lane some 25 instructions, waiting for the others costs the idle ones. 5e6 packages
// through the disk of 2.4e6 cells, 1, 2, 4, 8 and 12 cells: 3.85, 3.59, 3.25, 3.13 and 3.13
// ms (unrolled by two 3.21, which the grids beyond L2 gain from: 13.7 against 14.2 ms for
// 8.0e6 cells of four species); 7.3 to 5.3 warp instructions per crossing. With the
// path-length tally two: see pool_warp.
constexpr int kWalkSteps = 8, kTallySteps = 2;

enum Adv { kCrossed = 0, kInteract = 1, kEscaped = 2, kError = 3 };

template <typename R>
__device__ __forceinline__ void set_inverse(Pkg<R>& k) {
#pragma unroll
  for (int a = 0; a < 3; ++a) k.inv[a] = k.d[a] == (R)0 ? (R)INFINITY : (R)1 / k.d[a];
}

template <typename R>
__device__ __forceinline__ void emit(Pkg<R>& k, unsigned long long id, const DevRun& r,
                                     const float* star_cdf, int B) {
  uint4 w = draw(r.seed, id, 0u, 0u);
  k.id = id;
  k.event = 0;
  k.bin = search_cdf(star_cdf, B, unit<float>(w.x));
  if (r.source_kind == 1) {
#pragma unroll
    for (int a = 0; a < 3; ++a) k.d[a] = sizeof(R) == 8 ? (R)r.beam64[a] : (R)r.beam[a];
  } else {
    isotropic<R>(unit<R>(w.y), unit<R>(w.z), k.d);
  }
  k.tau = -log_(unit<R>(w.w));
#pragma unroll
  for (int a = 0; a < 3; ++a) k.p[a] = sizeof(R) == 8 ? (R)r.src64[a] : (R)r.src[a];
  set_inverse(k);
}

// One cell: cross it, or move to the interaction point inside it (the leaf is found
// from the base cube each time: the plain walk). kTally: path lengths into pathabs.
template <typename R, bool kTally>
__device__ __forceinline__ int advance(Pkg<R>& k, const DevGrid& g, const Kappa* kap,
                                       int& leaf, int& level, float* pathabs) {
  int I[3];
  int rc = locate(g, k.p, k.d, leaf, level, I);
  if (rc == 1) return kEscaped;
  if (rc < 0) return kError;
  const R sz = (R)1 / (R)(1 << level);
  const R lo0 = (R)I[0] * sz, lo1 = (R)I[1] * sz, lo2 = (R)I[2] * sz;
  const R hi0 = lo0 + sz, hi1 = lo1 + sz, hi2 = lo2 + sz;
  const R d0 = k.d[0], d1 = k.d[1], d2 = k.d[2];
  const R inf = (R)INFINITY;
  const R t0 = d0 > (R)0 ? (hi0 - k.p[0]) * k.inv[0] : (d0 < (R)0 ? (lo0 - k.p[0]) * k.inv[0] : inf);
  const R t1 = d1 > (R)0 ? (hi1 - k.p[1]) * k.inv[1] : (d1 < (R)0 ? (lo1 - k.p[1]) * k.inv[1] : inf);
  const R t2 = d2 > (R)0 ? (hi2 - k.p[2]) * k.inv[2] : (d2 < (R)0 ? (lo2 - k.p[2]) * k.inv[2] : inf);
  int ax;
  R tex;
  if (t0 <= t1 && t0 <= t2) {
    ax = 0;
    tex = t0;
  } else if (t1 <= t2) {
    ax = 1;
    tex = t1;
  } else {
    ax = 2;
    tex = t2;
  }
  tex = fmax(tex, (R)0);
  // extinction per base-cube unit of path: sum_s (rho_s d0) kappa_ext,s(bin)
  const float* rho = g.rho + (size_t)leaf * g.S;
  const Kappa* kb = kap + k.bin * g.S;
  R kx = (R)0;
  for (int s = 0; s < g.S; ++s) kx += (R)__ldg(&rho[s]) * (R)kb[s].kext;
  const R dtau = kx * tex;
  if constexpr (kTally) {  // path-length tally of the segment inside this cell
    const R seg = (kx > (R)0 && dtau > k.tau) ? k.tau / kx : tex;
    float* row = pathabs + tally_place(leaf) * tally_row(g.S);
    for (int s = 0; s < g.S; ++s) {
      const float v = (float)((R)__ldg(&rho[s]) * (R)kb[s].kabs * seg);
      if (v > 0.f) atomicAdd(row + s, v);
    }
  }
  if (kx > (R)0 && dtau > k.tau) {
    const R sd = k.tau / kx;
    k.p[0] = fmin(hi0, fmax(lo0, k.p[0] + sd * d0));
    k.p[1] = fmin(hi1, fmax(lo1, k.p[1] + sd * d1));
    k.p[2] = fmin(hi2, fmax(lo2, k.p[2] + sd * d2));
    return kInteract;
  }
  k.tau -= dtau;
  const R f0 = d0 > (R)0 ? hi0 : lo0, f1 = d1 > (R)0 ? hi1 : lo1, f2 = d2 > (R)0 ? hi2 : lo2;
  k.p[0] = ax == 0 ? f0 : fmin(hi0, fmax(lo0, k.p[0] + tex * d0));
  k.p[1] = ax == 1 ? f1 : fmin(hi1, fmax(lo1, k.p[1] + tex * d1));
  k.p[2] = ax == 2 ? f2 : fmin(hi2, fmax(lo2, k.p[2] + tex * d2));
  return kCrossed;
}

// ---------------------------------------------------------------- forward frame
// The pool's walks run in a frame in which the package moves forward along every axis:
// an axis with d < 0 is mirrored (p -> -p, d -> -d; a cell [lo, hi] -> [-hi, -lo]), which
// FP32 does exactly, and every operation of the walk commutes with the sign, so the
// positions are bit for bit those of the unmirrored walk. The face ahead is then always
// lo + edge, a position can only pass its cell's upper bound (one minimum instead of a
// clamp), the neighbour's corner is the face itself, and the child of a point is a plain
// floor. Pkg::p, d, inv and the cell's corner are kept mirrored between interactions;
// the frame changes with the direction (orient).
// Together with what moved out of the step (the move to an interaction point into the
// interaction phase, the spectrum of escaped packages into the refill, the rarer counters
// into shared memory) it took the linked walk on the disk of 2.4e6 cells from 11.5 to 8.3
// warp instructions per crossing and 5e6 packages from 5.08 to 4.17 ms at four blocks per
// SM; the path walk on 8.0e6 cells, 1e7 packages, from 22.8 to 22.1 ms.
//
// Pkg::dirs: bits 24-26, the mirrored axes; byte a (a = 0, 1, 2), what the walk looks up
// by the exit axis: linked, the byte offset of the face's link in the record; path, 0x80
// where the axis is mirrored.
__device__ __forceinline__ unsigned mirrored(const Pkg<float>& k) { return (k.dirs >> 24) & 7u; }

template <bool kPath, class CellT>
__device__ __forceinline__ void orient(Pkg<float>& k, CellT& c, unsigned was) {
  unsigned dirs = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const bool neg = k.d[a] < 0.f;
    if (neg != (((was >> a) & 1u) != 0u)) {
      k.p[a] = -k.p[a];
      c.lo[a] = -(c.lo[a] + c.sz);
    }
    k.d[a] = fabsf(k.d[a]);
    k.inv[a] = fabsf(k.inv[a]);
    if (neg) dirs |= 1u << (24 + a);
    if (kPath)
      dirs |= neg ? 0x80u << (8 * a) : 0u;
    else
      dirs |= (unsigned)(8 * a + (neg ? 0 : 4)) << (8 * a);
  }
  k.dirs = dirs;
}

// the direction with its signs back (k.d only), and one component of a position
__device__ __forceinline__ void restore_direction(Pkg<float>& k) {
#pragma unroll
  for (int a = 0; a < 3; ++a)
    if ((k.dirs >> (24 + a)) & 1u) k.d[a] = -k.d[a];
}

__device__ __forceinline__ float true_component(const Pkg<float>& k, float v, int a) {
  return (k.dirs >> (24 + a)) & 1u ? -v : v;
}

// What byte a of k.dirs says of the exit axis: for the linked walk the byte, for the path
// walk its top bit over all 32 bits. (prmt itself: the intrinsic for it ignores the
// selector bit that spreads the sign.)
__device__ __forceinline__ unsigned pick_byte(unsigned x, unsigned sel) {
  unsigned r;
  asm("prmt.b32 %0, %1, 0, %2;" : "=r"(r) : "r"(x), "r"(sel));
  return r;
}

// Distance to the nearest face ahead and its axis (the lowest on ties): ax0, ax1 or
// neither. An axis with d == 0 has inv = +inf and gives +inf, or NaN on its upper face,
// which the minimum never picks.
struct Exit {
  float F[3], t;
  bool ax0, ax1;
};

template <class CellT>
__device__ __forceinline__ Exit exit_of(const Pkg<float>& k, const CellT& c) {
  Exit e;
  float t[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    e.F[a] = c.lo[a] + c.sz;
    t[a] = (e.F[a] - k.p[a]) * k.inv[a];
  }
  e.t = fminf(fminf(t[0], t[1]), t[2]);
  e.ax0 = t[0] == e.t;
  e.ax1 = !e.ax0 && t[1] == e.t;
  return e;
}

// onto the face ahead; the corner becomes that of the same-size neighbour
template <class CellT>
__device__ __forceinline__ void cross(Pkg<float>& k, CellT& c, const Exit& e) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const bool here = a == 0 ? e.ax0 : (a == 1 ? e.ax1 : !(e.ax0 || e.ax1));
    const float v = fminf(e.F[a], fmaf(e.t, k.d[a], k.p[a]));
    k.p[a] = here ? e.F[a] : v;
    c.lo[a] = here ? e.F[a] : c.lo[a];
  }
}

// to the interaction point: tau spent inside the cell at extinction kx
template <class CellT>
__device__ __forceinline__ void to_point(Pkg<float>& k, const CellT& c, float kx) {
  const float sd = k.tau / kx;
#pragma unroll
  for (int a = 0; a < 3; ++a)
    k.p[a] = fminf(c.lo[a] + c.sz, fmaf(sd, k.d[a], k.p[a]));
}

// ---------------------------------------------------------------- linked walk
// The leaf a package is in, with its lower corner (in the package's forward frame) and
// its edge (base-cube units; both exact in FP32: multiples of 2^-level below 2^13).
struct Cell {
  int leaf;
  float lo[3];
  float sz;  // 2^-level
  __device__ __forceinline__ int level() const { return 127 - (__float_as_int(sz) >> 23); }
};

template <class CellT>
__device__ __forceinline__ void set_corner(CellT& c, const int I[3], int level) {
  c.sz = __int_as_float((127 - level) << 23);
#pragma unroll
  for (int a = 0; a < 3; ++a) c.lo[a] = (float)I[a] * c.sz;
}

// Enter the grid at the package's position (full descent from the base cube).
__device__ __forceinline__ int enter(Pkg<float>& k, const DevGrid& g, Cell& c,
                                     unsigned& child_reads) {
  int I[3], level;
  int rc = locate<float>(g, k.p, k.d, c.leaf, level, I);
  if (rc == 0) {
    child_reads += level;
    set_corner(c, I, level);
    orient<false>(k, c, 0u);
  }
  return rc;
}

// The densities of a leaf as one vector (kS = 2: from its face-link record, 4: from the
// density rows), and the sum of densities times a bin's opacities.
template <int kS>
__device__ __forceinline__ float4 leaf_rho(const DevGrid& g, int leaf) {
  if constexpr (kS == 2) {
    const float2 r = __ldg(reinterpret_cast<const float2*>(g.links + (size_t)leaf * kRec + 6));
    return make_float4(r.x, r.y, 0.f, 0.f);
  } else if constexpr (kS == 4) {
    return __ldg(reinterpret_cast<const float4*>(g.rho) + leaf);
  } else {
    return make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// A bin's opacities of kS species as one vector, from a table [B][kS].
template <int kS>
__device__ __forceinline__ float4 bin_vec(const float* table, int bin) {
  if constexpr (kS == 4) {
    return reinterpret_cast<const float4*>(table)[bin];
  } else if constexpr (kS == 2) {
    const float2 e = reinterpret_cast<const float2*>(table)[bin];
    return make_float4(e.x, e.y, 0.f, 0.f);
  } else {
    return make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// Extinction of a leaf per base-cube unit of path at a bin. kS: the species count when
// fixed at compile time (2 or 4: the densities r, the bin's opacities as one vector), 0 when
// read from the grid (densities from the face-link record for one or two species). The
// opacities come from kext [B][S]. kInOrder: the launches with the path-length tally, summed
// species by species as the generic form does (their histories are those of the generic walk
// to the last bit), the generic form's opacities from the records kap it reads anyway.
template <int kS, bool kInOrder = false>
__device__ __forceinline__ float leaf_ext(const DevGrid& g, int leaf, float4 r, int bin,
                                          const Kappa* kap, const float* kext) {
  if constexpr (kS == 2) {
    const float4 e = bin_vec<2>(kext, bin);
    if constexpr (kInOrder) return fmaf(r.y, e.y, r.x * e.x);
    return r.x * e.x + r.y * e.y;
  } else if constexpr (kS == 4) {
    const float4 e = bin_vec<4>(kext, bin);
    if constexpr (kInOrder)
      return fmaf(r.w, e.w, fmaf(r.z, e.z, fmaf(r.y, e.y, r.x * e.x)));
    return r.x * e.x + r.y * e.y + r.z * e.z + r.w * e.w;
  } else {
    const Kappa* kb = kap + bin * g.S;
    const float* eb = kext + bin * g.S;
    const auto e = [&](int s) { return kInOrder ? kb[s].kext : eb[s]; };
    if (g.S <= 2) {
      const int* rec = g.links + (size_t)leaf * kRec;
      float kx = __int_as_float(__ldg(rec + 6)) * e(0);
      if (g.S == 2) kx += __int_as_float(__ldg(rec + 7)) * e(1);
      return kx;
    }
    const float* rho = g.rho + (size_t)leaf * g.S;
    float kx = 0.f;
    for (int s = 0; s < g.S; ++s) kx += __ldg(&rho[s]) * e(s);
    return kx;
  }
}

// Vector additions to memory, left out where nothing is to be added.
__device__ __forceinline__ void red_add2(float* p, float v0, float v1) {
  if (v0 > 0.f || v1 > 0.f)
    asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(__cvta_generic_to_global(p)),
                 "f"(v0), "f"(v1)
                 : "memory");
}

__device__ __forceinline__ void red_add4(float* p, const float* v) {
  if (v[0] > 0.f || v[1] > 0.f || v[2] > 0.f || v[3] > 0.f)
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(
                     __cvta_generic_to_global(p)),
                 "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3])
                 : "memory");
}

// Path-length tallies of a segment of length seg in a leaf, in its row: rho_s kappa_abs,s seg is
// added for every species. With the species of a cell side by side two
// or four of them are one vector reduction to one sector. 2e6 packages through 1.06e6
// cells of two species: 3.9 ms with an atomic per species into arrays apart (and the
// generic species loop), 2.7 ms. Other species counts need rows of whole vectors: 1e6
// packages through 6.4e4 cells of three, five and eight species took 2.27, 2.83 and 5.06 ms
// with an array per species, 2.78, 3.96 and 5.32 with single atomics into rows of S, and 1.16,
// 1.78 and 3.57 so.
template <int kS>
__device__ __forceinline__ void tally_segment(const DevGrid& g, float* pathabs, int leaf,
                                              float4 r, int bin, float seg, const Kappa* kap,
                                              const float* kabs) {
  if constexpr (kS == 2) {
    const float4 a = bin_vec<2>(kabs, bin);
    red_add2(pathabs + 2 * tally_place(leaf), r.x * a.x * seg, r.y * a.y * seg);
  } else if constexpr (kS == 4) {
    const float4 a = bin_vec<4>(kabs, bin);
    const float v[4] = {r.x * a.x * seg, r.y * a.y * seg, r.z * a.z * seg, r.w * a.w * seg};
    red_add4(pathabs + 4 * tally_place(leaf), v);
  } else {
    const int S = g.S;
    const float* rho = g.rho + (size_t)leaf * S;
    const Kappa* kb = kap + bin * S;
    float* row = pathabs + tally_place(leaf) * tally_row(S);
    if (S == 1) {
      const float v = __ldg(rho) * kb[0].kabs * seg;
      if (v > 0.f) atomicAdd(row, v);
      return;
    }
    for (int s = 0; s < S; s += 4) {
      float v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = s + j < S ? __ldg(&rho[s + j]) * kb[s + j].kabs * seg : 0.f;
      if (S == 2)
        red_add2(row, v[0], v[1]);
      else
        red_add4(row + s, v);
    }
  }
}

// One cell of the walk using the face links: the exit face follows from the
// geometry alone, so the face link and the densities come from one record read;
// the next leaf is the linked one (same size or coarser), or is found by a short
// descent when the neighbouring region is finer. Where the optical depth runs out
// inside the cell nothing is changed (to_point follows in the interaction phase, which
// runs with more lanes). kLos: a sight line, which never interacts and adds the cell's
// optical depth to *tau_los instead. kTally: the path-length tallies, into pathabs (kabs:
// the absorption opacities [B][kS]).
template <bool kLos = false, int kS = 0, bool kTally = false>
__device__ __forceinline__ int advance_linked(Pkg<float>& k, Cell& c, const DevGrid& g,
                                              const Kappa* kap, const float* kext,
                                              unsigned& child_reads, float* tau_los = nullptr,
                                              float* pathabs = nullptr,
                                              const float* kabs = nullptr) {
  const Exit e = exit_of(k, c);
  const float4 r = leaf_rho<kS>(g, c.leaf);
  const float kx = leaf_ext<kS, kTally>(g, c.leaf, r, k.bin, kap, kext);
  const unsigned off =
      pick_byte(k.dirs, e.ax0 ? 0x4440u : (e.ax1 ? 0x4441u : 0x4442u));
  const int link = __ldg(reinterpret_cast<const int*>(
      reinterpret_cast<const char*>(g.links + (size_t)c.leaf * kRec) + off));
  const float dtau = kx * e.t;
  bool hit;
  if constexpr (kLos) {
    *tau_los += dtau;
    hit = false;
  } else {
    hit = dtau > k.tau;  // only where kx > 0
  }
  if constexpr (kTally)
    tally_segment<kS>(g, pathabs, c.leaf, r, k.bin, hit ? k.tau / kx : e.t, kap, kabs);
  if (hit) return kInteract;
  if constexpr (!kLos) k.tau -= dtau;
  cross(k, c, e);
  if ((unsigned)link < (unsigned)kLinkSame) {  // a leaf of the same size
    c.leaf = link;
    return kCrossed;
  }
  if (link >= 0) {  // a leaf of the same size or coarser: round the corner down to its edge
    c.leaf = link & kLinkLeafMask;
    const int bits = __float_as_int(c.sz) + ((link >> 28) << 23);
    c.sz = __int_as_float(bits);
    // exact: adding 1.5 * 2^23 edges (corners lie below 2^18 of them) leaves multiples of one
    const float big = __int_as_float(bits + (23 << 23) + (1 << 22));
#pragma unroll
    for (int a = 0; a < 3; ++a) c.lo[a] = __fadd_rd(c.lo[a], big) - big;
    return kCrossed;
  }
  if (link == kLinkEscape) return kEscaped;
  // the same-size neighbour is split: descend, staying inside that node (on the side of
  // each middle that the position is on). A step of a warp has a lane here more often than
  // not, so this is kept short: in integers with conversions, and floorf above, 5e6
  // packages through the disk took 3.93 ms against 3.85.
  int code = link, left = g.max_level - c.level();
  float h = c.sz;
  for (;;) {
    const int blk = -code - 1;
    if (blk >= g.n_blocks || left-- <= 0) return kError;
    ++child_reads;
    h *= 0.5f;
    unsigned oct = mirrored(k);  // a mirrored axis numbers its children backwards
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float mid = c.lo[a] + h;
      if (k.p[a] >= mid) {
        c.lo[a] = mid;
        oct ^= 1u << a;
      }
    }
    code = __ldg(&g.child[(size_t)blk * 8 + oct]);
    if (code >= 0) {
      if ((long long)code >= g.n_leaves) return kError;
      c.leaf = code;
      c.sz = h;
      return kCrossed;
    }
  }
}

// ---------------------------------------------------------------- path walk
// The walk without face links. A package keeps the ids of the child blocks on the
// path from its base cube to its leaf (blk(l): the block holding the path's node at
// level l). Crossing a face, it climbs to the deepest common ancestor of its leaf and
// of the neighbouring position -- the highest bit in which their integer coordinates
// differ gives the number of levels to climb -- and descends from there: a neighbour
// in the same block costs one child read, in the sector the leaf's own read left in
// L1. Its random reads go to the densities and the child table (3.5 GB for the large
// disk's 1.7e8 cells) instead of the face-link records and densities (8.3 GB), whose
// address translation misses cost more than the extra reads on grids that large. The
// geometry is the linked walk's, and so is every neighbour it finds: both walks give
// the same histories.
constexpr int kPathLevels = 4;  // the path walk serves grids of at most 4 levels

struct PathCell {
  int slot;     // tree slot of the leaf: its row in rho_slot
  float kx;     // the leaf's extinction at the package's bin
  float lo[3];  // lower corner, in the package's forward frame
  float sz;     // 2^-level
  int b0;       // base cube the package is in
  int b1, b2, b3, b4;
  __device__ __forceinline__ int level() const { return 127 - (__float_as_int(sz) >> 23); }
  __device__ __forceinline__ int blk(int l) const {
    return l == 1 ? b1 : (l == 2 ? b2 : (l == 3 ? b3 : b4));
  }
  __device__ __forceinline__ void set_blk(int l, int b) {
    if (l == 1) b1 = b;
    else if (l == 2) b2 = b;
    else if (l == 3) b3 = b;
    else b4 = b;
  }
};

// Enter the grid at the package's position: descent from the base cube, recording
// the blocks on the path. 0 inside, 1 outside, -1 malformed (or deeper than the
// walk serves).
__device__ __forceinline__ int enter_path(Pkg<float>& k, const DevGrid& g, PathCell& c,
                                          unsigned& child_reads) {
  const int n = g.n_base;
  int I[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    I[a] = cell_index(k.p[a], k.d[a]);
    if (I[a] < 0 || I[a] >= n) return 1;
  }
  int slot = I[0] + n * (I[1] + n * I[2]);
  c.b0 = slot;
  int node = __ldg(&g.base[slot]);
  int lev = 0;
  while (node < 0) {
    const long long blk = -(long long)node - 1;
    if (blk >= g.n_blocks || lev >= g.max_level || lev >= kPathLevels) return -1;
    ++lev;
    c.set_blk(lev, (int)blk);
    const float sc = (float)(1 << lev);
    int oct = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int j = cell_index(k.p[a] * sc, k.d[a]);
      const int o = j - 2 * I[a];
      if ((unsigned)o > 1u) return -1;
      oct |= o << a;
      I[a] = j;
    }
    slot = g.n_base3 + (int)blk * 8 + oct;
    node = __ldg(&g.child[blk * 8 + oct]);
    ++child_reads;
  }
  if ((long long)node >= g.n_leaves) return -1;
  c.slot = slot;
  set_corner(c, I, lev);
  orient<true>(k, c, 0u);
  return 0;
}

// The row of a tree slot as one vector (kS = 4 or 2 species; the generic form reads
// the first word here and the rest in slot_ext): a leaf's densities, or for a refined
// slot the child block's code -(block + 1) in the first word (densities are >= +0, so
// the sign bit tells them apart); and the extinction sum over species at the bin's
// opacities kb.
template <int kS>
__device__ __forceinline__ float4 slot_row(const DevGrid& g, int slot) {
  if constexpr (kS == 4) {
    return __ldg(reinterpret_cast<const float4*>(g.rho_slot) + slot);
  } else if constexpr (kS == 2) {
    const float2 v = __ldg(reinterpret_cast<const float2*>(g.rho_slot) + slot);
    return make_float4(v.x, v.y, 0.f, 0.f);
  } else {
    return make_float4(__ldg(&g.rho_slot[(size_t)slot * g.S]), 0.f, 0.f, 0.f);
  }
}

// The leaf id of a leaf's tree slot (from the tree arrays; the walk itself reads only
// the rows), or -1 if the slot holds no leaf.
__device__ __forceinline__ int path_leaf(const DevGrid& g, int slot) {
  const int node = slot < g.n_base3 ? __ldg(&g.base[slot]) : __ldg(&g.child[slot - g.n_base3]);
  return node >= 0 && (long long)node < g.n_leaves ? node : -1;
}

template <int kS>
__device__ __forceinline__ float slot_ext(const DevGrid& g, float4 v, int slot, float4 e,
                                          const float* eb) {
  if constexpr (kS == 4) {
    return v.x * e.x + v.y * e.y + v.z * e.z + v.w * e.w;
  } else if constexpr (kS == 2) {
    return v.x * e.x + v.y * e.y;
  } else {
    const float* rho = g.rho_slot + (size_t)slot * g.S;
    float kx = 0.f;
    for (int s = 0; s < g.S; ++s) kx += __ldg(&rho[s]) * eb[s];
    return kx;
  }
}

// The extinction of the cell a package is in, at its bin.
template <int kS>
__device__ __forceinline__ float path_ext(const DevGrid& g, int slot, int bin,
                                          const float* kext) {
  return slot_ext<kS>(g, slot_row<kS>(g, slot), slot, bin_vec<kS>(kext, bin),
                      kext + bin * (kS > 0 ? kS : g.S));
}

// One cell of the path walk (kS: 2 or 4 species read as one vector, 0 the generic
// loop). The next cell is found from the rows alone: the slot of the first node off
// the package's path is known from the block ids it carries (the next base cube is a
// stride away from its own), and that slot's row is either the leaf's densities or the
// code of the block to descend into -- one read per crossing (one more per level
// descended). Integer coordinates are formed only in refined cubes; between base cubes,
// most of a large grid's crossings, there are none. The extinction at the package's bin
// is kept in the cell for the next step.
template <int kS>
__device__ __forceinline__ int advance_path(Pkg<float>& k, PathCell& c, const DevGrid& g,
                                            const float* kext, unsigned& child_reads) {
  const Exit e = exit_of(k, c);
  const float dtau = c.kx * e.t;
  if (dtau > k.tau) return kInteract;
  k.tau -= dtau;
  const float Fax = e.ax0 ? e.F[0] : (e.ax1 ? e.F[1] : e.F[2]);
  const int n = g.n_base;
  // all ones where the exit axis is mirrored: the domain then ends at 0 and the base
  // cubes' numbers fall
  const int m = (int)pick_byte(k.dirs, e.ax0 ? 0x8888u : (e.ax1 ? 0x9999u : 0xAAAAu));
  if (Fax >= __int_as_float(__float_as_int((float)n) & ~m)) return kEscaped;
  cross(k, c, e);
  const int stride = e.ax0 ? 1 : (e.ax1 ? n : n * n);
  const int next = c.b0 + (stride ^ m) - m;
  const float sz = c.sz;
  int slot = next, lev = 0, L = 0;
  int J[3];
  if (sz != 1.f) {
    L = c.level();
    const float iz = __int_as_float((127 + L) << 23);
#pragma unroll
    for (int a = 0; a < 3; ++a) J[a] = (int)(c.lo[a] * iz);
    const int Jax = (int)(Fax * iz);
    const int u = 32 - __clz(Jax ^ (Jax - 1));  // levels up to the common ancestor
    if (u <= L) {  // the common ancestor's block holds the first node off the path
      lev = L - u + 1;
      const int sh = L - lev;
      const unsigned oct = (unsigned)(((J[0] >> sh) & 1) | (((J[1] >> sh) & 1) << 1) |
                                      (((J[2] >> sh) & 1) << 2)) ^ mirrored(k);
      slot = g.n_base3 + c.blk(lev) * 8 + (int)oct;
    }
  }
  if (lev == 0) c.b0 = next;
  float4 row = slot_row<kS>(g, slot);
  int code = __float_as_int(row.x);
  if (sz != 1.f || code < 0) {
    if (sz == 1.f) {
#pragma unroll
      for (int a = 0; a < 3; ++a) J[a] = (int)c.lo[a];
    }
    int K[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) K[a] = J[a] >> (L - lev);
    while (code < 0) {
      const long long blk = -(long long)code - 1;
      if (blk >= g.n_blocks || lev >= g.max_level || lev >= kPathLevels) return kError;
      ++lev;
      c.set_blk(lev, (int)blk);
      unsigned oct = mirrored(k);
      if (lev <= L) {
#pragma unroll
        for (int a = 0; a < 3; ++a) K[a] = J[a] >> (L - lev);
      } else {  // a finer neighbour: the child holding the crossing point
        const float sc = __int_as_float((127 + lev) << 23);
#pragma unroll
        for (int a = 0; a < 3; ++a)
          K[a] = min(max(__float2int_rd(k.p[a] * sc), 2 * K[a]), 2 * K[a] + 1);
      }
#pragma unroll
      for (int a = 0; a < 3; ++a) oct ^= (unsigned)(K[a] & 1) << a;
      slot = g.n_base3 + (int)blk * 8 + (int)oct;
      row = slot_row<kS>(g, slot);
      code = __float_as_int(row.x);
      ++child_reads;
    }
    set_corner(c, K, lev);
  }
  c.slot = slot;
  c.kx = slot_ext<kS>(g, row, slot, bin_vec<kS>(kext, k.bin), kext + k.bin * (kS > 0 ? kS : g.S));
  return kCrossed;
}

constexpr float kInv4Pi = 0.0795774715459476679f;  // 1 / (4 pi)

// Henyey-Greenstein phase function per steradian at cos(angle) = mu.
__device__ __forceinline__ float hg_per_sr(float g, float mu) {
  const float den = fmaxf(1.f + g * g - 2.f * g * mu, 1e-30f);
  return (1.f - g * g) * kInv4Pi / (den * sqrtf(den));
}

// Interaction part 1: draw the event's numbers; scatter completely, or pick the
// absorbing species. Returns the species (>= 0) for an absorption, -1 for a scatter.
// peel_o / peel_w (peel-off): for a scattering, *peel_w receives the phase function
// per steradian toward the unit vector peel_o, at the direction before the turn.
// kS: the species count when fixed at compile time (2: the densities come from the
// cell's face-link record, which the linked walk has just read; -2 or -4: from the
// slot row, which the path walk has just read), 0 when read from the grid. `row` is
// the leaf id, or for the path walk (kS < 0) the leaf's tree slot.
template <int kS>
__device__ __forceinline__ float cell_rho(const DevGrid& g, int row, int s) {
  if (kS == 2) return __int_as_float(__ldg(g.links + (size_t)row * kRec + 6 + s));
  if (kS < 0) return __ldg(&g.rho_slot[(size_t)row * (size_t)(kS < 0 ? -kS : 1) + s]);
  return __ldg(&g.rho[(size_t)row * g.S + s]);
}

template <typename R, int kS = 0>
__device__ __forceinline__ int interact(Pkg<R>& k, const DevGrid& g, const Kappa* kap,
                                        int row, const DevRun& r, uint4& w1,
                                        const float* peel_o = nullptr,
                                        float* peel_w = nullptr) {
  uint4 w0 = draw(r.seed, k.id, k.event, 0u);
  w1 = draw(r.seed, k.id, k.event, 1u);
  const int S = kS > 0 ? kS : (kS < 0 ? -kS : g.S);
  const Kappa* kb = kap + k.bin * S;
  float ksca = 0.f, kext = 0.f, kabs = 0.f;
  for (int s = 0; s < S; ++s) {
    const float rs = cell_rho<kS>(g, row, s);
    ksca += rs * kb[s].ksca;
    kext += rs * kb[s].kext;
    kabs += rs * kb[s].kabs;
  }
  const float xs = unit<float>(w0.y);
  int sp = S - 1;
  if (unit<float>(w0.x) * kext < ksca) {
    const float target = xs * ksca;
    float cum = 0.f;
    for (int s = 0; s < S; ++s) {
      cum += cell_rho<kS>(g, row, s) * kb[s].ksca;
      if (cum > target) { sp = s; break; }
    }
    if (peel_w)
      *peel_w = hg_per_sr(kb[sp].g, (float)k.d[0] * peel_o[0] + (float)k.d[1] * peel_o[1] +
                                        (float)k.d[2] * peel_o[2]);
    R mu = hg_mu<R>((R)kb[sp].g, unit<R>(w0.z));
    turn<R>(k.d, mu, unit<R>(w0.w));
    set_inverse(k);
    k.tau = -log_(unit<R>(w1.x));
    return -1;
  }
  const float target = xs * kabs;
  float cum = 0.f;
  for (int s = 0; s < S; ++s) {
    cum += cell_rho<kS>(g, row, s) * kb[s].kabs;
    if (cum > target) { sp = s; break; }
  }
  isotropic<R>(unit<R>(w0.z), unit<R>(w0.w), k.d);
  set_inverse(k);
  k.tau = -log_(unit<R>(w1.x));
  return sp;
}

// Interaction part 2 (absorption): n is this package's place in the cell's
// absorption count (the count before it); draw the new bin.
template <typename R, int kS = 0>
__device__ __forceinline__ void reemit(Pkg<R>& k, const DevGrid& g, const DevTables& t,
                                       const DevRun& r, int s, int leaf, int row, int level,
                                       unsigned long long n, const uint4& w1,
                                       unsigned& clamped) {
  float xu = unit<float>(w1.y), xb = unit<float>(w1.z);
  float rho = cell_rho<kS>(g, row, s);
  float u;
  if (r.mode == 0) {
    float e = r.count_scale * t.eps_d0_over_V[level] / rho;
    u = ((float)n + xu) * e;
  } else if (r.mode == 1) {
    float e = r.count_scale * t.eps_d0_over_V[level] / rho;
    u = xu * fmaxf((float)n * e, t.u_tmin[s]);
  } else {
    u = xu * __ldg(&t.u_frozen[(size_t)s * g.n_leaves + leaf]);
  }
  const float* S = t.S32 + (size_t)s * g.n_T;
  int nI = g.n_T - 1;
  int i;
  if (u >= __ldg(&S[nI])) {
    i = nI - 1;
    ++clamped;
  } else {
    // interval i with S[i] <= u < S[i+1]: start from the guide, finish by scanning
    float kf = (__logf(fmaxf(u, 1e-30f)) - t.u_ln0[s]) * t.u_inv[s];
    int kk = (int)fminf(fmaxf(kf, 0.0f), (float)nI);
    i = __ldg(&t.u_guide[s * g.n_T + kk]);
    while (i > 0 && __ldg(&S[i]) > u) --i;
    while (i + 1 < nI && __ldg(&S[i + 1]) <= u) ++i;
  }
  // first bin whose cumulative value exceeds xb: guide start, then scan
  const size_t cdf_row = ((size_t)s * nI + i) * g.B;
  const float* cdf = t.dcdf + cdf_row;
  int b = __ldg(&t.cdf_guide[cdf_row + min((int)(xb * (float)g.B), g.B - 1)]);
  while (b > 0 && __ldg(&cdf[b - 1]) > xb) --b;
  while (__ldg(&cdf[b]) <= xb) ++b;
  k.bin = b;
}

// New bin after an absorption by PAH number p: drawn from the PAH's emission
// spectrum in this cell (its template unless a per-cell spectrum is set).
template <typename R>
__device__ __forceinline__ void pah_bin(Pkg<R>& k, const DevGrid& g, const DevTables& t, int p,
                                        int leaf, const uint4& w1) {
  const float xb = unit<float>(w1.z);
  const float* cdf = t.pah_cdf + (size_t)p * g.B;
  if (t.pah_cell_cdf) {
    const float* cc = t.pah_cell_cdf + ((size_t)p * g.n_leaves + leaf) * g.B;
    if (__ldg(&cc[g.B - 1]) > 0.f) cdf = cc;
  }
  int lo = 0, hi = g.B - 1;
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (__ldg(&cdf[mid]) > xb) hi = mid; else lo = mid + 1;
  }
  k.bin = lo;
}

// Absorption by a PAH species: tally the photon in the cell's coarse absorbed
// spectrum and mark the cell as PAH-active for that PAH, then draw the new bin.
template <typename R>
__device__ __forceinline__ void pah_absorb(Pkg<R>& k, const DevGrid& g, const DevTables& t,
                                           const DevRun& r, int p, int leaf, const uint4& w1) {
  const int kc = (k.bin * t.n_coarse) / g.B;
  atomicAdd(&r.pahabs[((size_t)p * g.n_leaves + leaf) * t.n_coarse + kc], 1u);
  atomicOr(&r.pah_flag[leaf], 1u << p);
  pah_bin(k, g, t, p, leaf, w1);
}

__device__ __forceinline__ int dir_bin(float dz, int n_dir) {
  int b = (int)floorf(0.5f * (dz + 1.0f) * (float)n_dir);
  return min(max(b, 0), n_dir - 1);
}

__device__ __forceinline__ void flush_tally(Tally& tl, unsigned long long* c) {
  const unsigned v[kNumCounters] = {tl.emitted,   tl.escaped, tl.capped,
                                    tl.absorptions, tl.scatters, tl.crossings,
                                    tl.errors,    tl.clamped, tl.levels,
                                    tl.peel_events, tl.peel_crossings};
#pragma unroll
  for (int i = 0; i < kNumCounters; ++i) {
    unsigned long long x = v[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    if ((threadIdx.x & 31) == 0 && x) atomicAdd(&c[i], x);
  }
  tl = Tally{};
}

__device__ __forceinline__ void flush_warp(LaneTally& tl, unsigned* wt, unsigned long long* c) {
  const int lane = threadIdx.x & 31;
  unsigned long long cr = tl.crossings, lv = tl.levels;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    cr += __shfl_xor_sync(kFull, cr, o);
    lv += __shfl_xor_sync(kFull, lv, o);
  }
  __syncwarp();
  if (lane < kNumCounters) {
    const unsigned long long x =
        lane == kCCrossings ? cr : (lane == kCLevels ? lv : (unsigned long long)wt[lane]);
    if (x) atomicAdd(&c[lane], x);
    wt[lane] = 0;
  }
  __syncwarp();
  tl = LaneTally{};
}

// ---------------------------------------------------------------- peel-off
// Sight line from the point x (base-cube units) toward the observer at bin `bin`:
// the pixel x projects to and the attenuation exp(-tau) to the boundary. Returns
// false when x falls outside the image, tau passes pe.tau_max, or the walk fails
// (then the tree status bit is set).
__device__ __forceinline__ bool sight_line(const DevGrid& g, const float* kext,
                                           const DevPeel& pe, float x0, float x1, float x2,
                                           int bin, float& att, size_t& pix,
                                           unsigned& crossings, unsigned* status) {
  const float r0 = x0 - pe.centre, r1 = x1 - pe.centre, r2 = x2 - pe.centre;
  const float u = r0 * pe.e1[0] + r1 * pe.e1[1] + r2 * pe.e1[2];
  const float v = r0 * pe.e2[0] + r1 * pe.e2[1] + r2 * pe.e2[2];
  const int px = (int)floorf(u * pe.sx + 0.5f * (float)pe.nx);
  const int py = (int)floorf(v * pe.sy + 0.5f * (float)pe.ny);
  const int plane = __ldg(&pe.plane_of_bin[bin]);
  if (plane < 0 || px < 0 || px >= pe.nx || py < 0 || py >= pe.ny) return false;
  Pkg<float> k;
  k.p[0] = x0;
  k.p[1] = x1;
  k.p[2] = x2;
  k.d[0] = pe.o[0];
  k.d[1] = pe.o[1];
  k.d[2] = pe.o[2];
  set_inverse(k);
  k.bin = bin;
  k.tau = 0.f;
  Cell c;
  unsigned lv = 0;
  float tau = 0.f;
  const int rc = enter(k, g, c, lv);
  if (rc < 0) {
    atomicOr(status, kStatusTree);
    return false;
  }
  if (rc == 0) {
    // a straight line crosses at most 3 n 2^L finest cells of the n^3 base grid
    const long long cap = 3ll * ((long long)g.n_base << g.max_level) + 8;
    for (long long i = 0;; ++i) {
      const int a = advance_linked<true>(k, c, g, nullptr, kext, lv, &tau);
      ++crossings;
      if (a == kEscaped) break;
      if (a == kError || i >= cap) {
        atomicOr(status, kStatusTree);
        return false;
      }
      if (tau > pe.tau_max) return false;
    }
  }
  att = expf(-tau);
  pix = ((size_t)plane * pe.ny + py) * pe.nx + px;
  return true;
}

// Point-source emissions: all start at the source, so each bin's emissions of the
// launch are peeled together, then its count is cleared.
__global__ void k_peel_source(DevGrid g, DevTables t, DevRun r, DevPeel pe) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= g.B) return;
  const unsigned long long n = pe.n_emit[b];
  if (n == 0) return;
  pe.n_emit[b] = 0;
  if (r.source_kind == 1) return;
  float att;
  size_t pix;
  unsigned cr = 0;
  if (sight_line(g, t.kext, pe, r.src[0], r.src[1], r.src[2], b, att, pix, cr, r.status))
    atomicAdd(&pe.image[pix], (double)n * (double)kInv4Pi * (double)att);
  if (cr) atomicAdd(&r.counters[kCPeelCrossings], (unsigned long long)cr);
}

// The events a transport launch recorded: one sight line per thread (grid-stride).
// Events beyond the buffer's capacity were not recorded; their number is added to
// the dropped counter.
__global__ void __launch_bounds__(256) k_peel_trace(DevGrid g, DevTables t, DevRun r,
                                                    const __grid_constant__ DevPeel pe) {
  const unsigned long long n_rec = *pe.n_ev;
  const unsigned long long n = n_rec < pe.capacity ? n_rec : pe.capacity;
  if (blockIdx.x == 0 && threadIdx.x == 0 && n_rec > n)
    atomicAdd(&r.counters[kCPeelDropped], n_rec - n);
  unsigned cr = 0;
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
       i += (unsigned long long)gridDim.x * blockDim.x) {
    const float4 e = pe.ev[i];
    const int bin = pe.ev_bin[i];
    float att;
    size_t pix;
    if (sight_line(g, t.kext, pe, e.x, e.y, e.z, bin, att, pix, cr, r.status))
      atomicAdd(&pe.image[pix], (double)(e.w * att));
  }
  unsigned long long x = cr;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
  if ((threadIdx.x & 31) == 0 && x) atomicAdd(&r.counters[kCPeelCrossings], x);
}

__global__ void k_image_out(const double* image, long long n, double scale, double* out) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) out[i] = image[i] * scale;
}

// Mean over the rows whose centres lie within half_rows pixels of the image's
// centre line (|py + 1/2 - ny/2| <= half_rows) of plane a minus plane b (b < 0:
// none), times scale; one thread per column.
__global__ void k_image_profile(const double* image, int nx, int ny, int plane_a, int plane_b,
                                int half_rows, double scale, double* out) {
  const int px = blockIdx.x * blockDim.x + threadIdx.x;
  if (px >= nx) return;
  double sum = 0.0;
  int rows = 0;
  for (int py = 0; py < ny; ++py) {
    if (fabs(py + 0.5 - 0.5 * ny) > (double)half_rows) continue;
    double v = image[((size_t)plane_a * ny + py) * nx + px];
    if (plane_b >= 0) v -= image[((size_t)plane_b * ny + py) * nx + px];
    sum += v;
    ++rows;
  }
  out[px] = rows ? sum * scale / rows : 0.0;
}

// ---------------------------------------------------------------- plain kernel
// One thread per package, tables read from global memory, one global atomic per
// absorption and per escape. FP32 is held to 64 registers for four blocks per SM: with the 80
// the compiler takes by itself 4e6 packages through the disk of 1.9e7 cells took 28.2 ms, with
// 64 21.6.
template <typename R, bool kTally>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 4 : 2) k_transport_plain(DevGrid g, DevTables t, DevRun r) {
  Tally tl = {};
  unsigned long long idx = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
  const unsigned long long t0 = global_ns();
  if (idx < r.n_packages) {
    Pkg<R> k;
    emit<R>(k, r.first_id + idx, r, t.star_cdf, g.B);
    ++tl.emitted;
    unsigned steps = 0;
    for (;;) {
      if ((++steps & 1023u) == 0 && global_ns() - t0 > r.budget_ns) {
        atomicOr(r.status, kStatusTimeout);
        break;
      }
      int leaf, level;
      int a = advance<R, kTally>(k, g, t.kap, leaf, level, r.pathabs);
      if (a <= kInteract) tl.levels += level;
      if (a == kCrossed) { ++tl.crossings; continue; }
      if (a == kEscaped) {
        ++tl.escaped;
        int db = dir_bin((float)k.d[2], g.n_dir);
        atomicAdd(&r.sed[(size_t)db * g.B + k.bin], 1ull);
        if (k.event == 0) atomicAdd(&r.sed[(size_t)(g.n_dir + db) * g.B + k.bin], 1ull);
        break;
      }
      if (a == kError) {
        ++tl.errors;
        atomicOr(r.status, kStatusTree);
        break;
      }
      if (++k.event > r.max_events) { ++tl.capped; break; }
      uint4 w1;
      int s = interact<R>(k, g, t.kap, leaf, r, w1);
      if (s < 0) { ++tl.scatters; continue; }
      unsigned long long n = atomicAdd(&r.count[(size_t)s * g.n_leaves + leaf], 1ull);
      if (t.pah_of[s] >= 0)
        pah_absorb<R>(k, g, t, r, t.pah_of[s], leaf, w1);
      else
        reemit<R>(k, g, t, r, s, leaf, leaf, level, n, w1, tl.clamped);
      ++tl.absorptions;
    }
  }
  flush_tally(tl, r.counters);
}

// ---------------------------------------------------------------- pool loop
// Where a warp's package indices come from: one counter of the launch (one model), or
// the counter of the model the warp works on (a batch). take() gives the lane of rank
// `rank` among the warp's nd dead lanes its index; indices at or beyond the end mean that
// there is none left.
struct GlobalIds {
  unsigned long long* next;
  __device__ __forceinline__ unsigned long long take(int nd, int rank, int lane, int leader) {
    unsigned long long b = 0;
    if (lane == leader) b = atomicAdd(next, (unsigned long long)nd);
    return __shfl_sync(kFull, b, leader) + (unsigned long long)rank;
  }
};

// Reserves `chunk` >= 32 indices at a time, [pos, pos + left) being what remains of the
// warp's reservation.
struct ModelIds {
  unsigned long long* next;
  unsigned long long pos, end;  // end: the model's number of packages
  int left, chunk;
  __device__ __forceinline__ unsigned long long take(int nd, int rank, int lane, int leader) {
    unsigned long long j = pos + (unsigned long long)rank;
    if (nd <= left) {
      pos += (unsigned long long)nd;
      left -= nd;
      return j;
    }
    unsigned long long b = end;
    if (pos < end) {  // until a reservation came back empty
      if (lane == leader) b = atomicAdd(next, (unsigned long long)chunk);
      b = __shfl_sync(kFull, b, leader);
    }
    if (rank >= left) j = b + (unsigned long long)(rank - left);
    pos = b + (unsigned long long)(nd - left);
    left = chunk - (nd - left);
    return j;
  }
};

// ---------------------------------------------------------------- parked packages
// kPlaces places per warp in shared memory for packages that no lane is walking: a vector of
// 16 bytes per place and part, so that lanes using neighbouring places never conflict.
// Parts 0-3: position and tau; direction and bin; event, id, dirs and level; leaf and
// corner. The path walk adds its block ids (part 4) and, in 8 bytes, the last of them and
// the leaf's extinction. The reciprocals of the direction are computed again.
constexpr int kPlaces = 32;

template <bool kPath>
__host__ __device__ constexpr int park_bytes() {  // per warp (bound schedule: none)
  return kPlaces * (kPath ? 16 * 5 + 8 : 16 * 4);
}

__device__ __forceinline__ uint4 park_pack(int v, const Pkg<float>& k, int leaf, const float lo[3],
                                           int level) {
  const auto u = [](float x) { return (unsigned)__float_as_int(x); };
  if (v == 0) return make_uint4(u(k.p[0]), u(k.p[1]), u(k.p[2]), u(k.tau));
  if (v == 1) return make_uint4(u(k.d[0]), u(k.d[1]), u(k.d[2]), (unsigned)k.bin);
  if (v == 2)
    return make_uint4(k.event, (unsigned)k.id, (unsigned)(k.id >> 32),
                      k.dirs | (unsigned)level << 27);
  return make_uint4((unsigned)leaf, u(lo[0]), u(lo[1]), u(lo[2]));
}

// A lane's package to place `dst` (store) and place `src` to the lane (load); places left
// by loading lanes may be among those stored to.
template <bool kPath, class CellT>
__device__ __forceinline__ void park_exchange(uint4* park, Pkg<float>& k, CellT& c, bool load,
                                              int src, bool store, int dst) {
  const auto f = [](unsigned x) { return __int_as_float((int)x); };
#pragma unroll
  for (int v = 0; v < (kPath ? 6 : 4); ++v) {
    uint4 x = make_uint4(0, 0, 0, 0), y = x;
    uint2* last = reinterpret_cast<uint2*>(park + 5 * kPlaces);
    if (load) {
      if (v < 5) {
        x = park[v * kPlaces + src];
      } else {
        const uint2 w = last[src];
        x.x = w.x;
        x.y = w.y;
      }
    }
    __syncwarp();
    if constexpr (kPath) {
      if (v < 4) y = park_pack(v, k, c.slot, c.lo, c.level());
      else if (v == 4) y = make_uint4(c.b0, c.b1, c.b2, c.b3);
      else y = make_uint4(c.b4, (unsigned)__float_as_int(c.kx), 0, 0);
    } else {
      y = park_pack(v, k, c.leaf, c.lo, c.level());
    }
    if (store) {
      if (v < 5)
        park[v * kPlaces + dst] = y;
      else
        last[dst] = make_uint2(y.x, y.y);
    }
    if (load) {
      if (v == 0) {
        k.p[0] = f(x.x), k.p[1] = f(x.y), k.p[2] = f(x.z), k.tau = f(x.w);
      } else if (v == 1) {
        k.d[0] = f(x.x), k.d[1] = f(x.y), k.d[2] = f(x.z), k.bin = (int)x.w;
      } else if (v == 2) {
        k.event = x.x;
        k.id = (unsigned long long)x.z << 32 | x.y;
        k.dirs = x.w & 0x07ffffffu;
      } else if (v == 3) {
        c.lo[0] = f(x.y), c.lo[1] = f(x.z), c.lo[2] = f(x.w);
        if constexpr (kPath) c.slot = (int)x.x;
        else c.leaf = (int)x.x;
      }
      if constexpr (kPath) {
        if (v == 4) c.b0 = (int)x.x, c.b1 = (int)x.y, c.b2 = (int)x.z, c.b3 = (int)x.w;
        if (v == 5) c.b4 = (int)x.x, c.kx = f(x.y);
      }
    }
    // the level travels in part 2, the edge it gives is read by the packing above
    if (v == 2 && load) c.sz = __int_as_float((int)(127u - (x.w >> 27)) << 23);
  }
  __syncwarp();
}

// One warp of the packet pool. Lanes walk; a lane whose package reaches its interaction
// point or leaves the domain is idle. Once `batch` lanes are idle (or none walks) the warp
// finds them work, the first of these that applies:
//  - 32 packages wait for their interaction, in lanes or parked: all lanes take one
//    (walking packages are parked as ready) and the long, divergent interaction code runs
//    with a full warp; afterwards every lane walks on with what it has;
//  - packages are parked ready to walk: idle lanes take them, waiting ones are parked;
//  - the source is not dry: waiting packages are parked, the idle lanes filled with new ones;
//  - near the end of the source: interactions as soon as `batch` packages wait.
// batch: half of `interaction_batch` (8: 4 idle lanes of 32). Each package's history is
// unchanged by this schedule. With a package bound to its lane (waiting in place for eight
// others, dead lanes refilled every 32 steps) half of the lanes idled, and the interaction
// code ran with a quarter of them. Bound and parked, both walking eight cells at a time, ms:
// disk of 2.4e6 cells, 5e6 packages 3.45 and 3.21; 8.0e6 cells of four species, 1e7
// packages 15.4 and 13.7; disk with images 1.41 and 1.22; 24 models in a batch 6.44 and
// 5.87; 1e5 packages in a small sphere 0.083 and 0.085. (Bound and one cell at a time: 4.06,
// 17.7, 1.66, 7.09, 0.090.) 8, 16, 24 and 32 places, one cell at a time: 4.41, 4.09, 3.90
// and 3.85 ms for the disk; 2 KB a warp for 32 still leave L1 most of its room.
//
// kTally: packages stay bound to their lanes, dead lanes are refilled every `refill_period`
// rounds and `interaction_batch` lanes start an interaction phase. An FP32 tally of a cell
// that 1e5 packages cross loses increments below half a unit of its last place (1e-3 of a
// sum next to the source) unless the lanes that cross it together are combined first, as
// they are when they start together: the parked schedule would change that sum by 1e-4 of
// it. The tally's reductions bound these launches anyway (2.60 parked, 2.67 ms bound).
// Absorptions of lanes hitting the same (species, cell) in one phase are merged into
// one atomic. `sed` is the escaped-spectrum histogram (shared or global memory).
// kPeel: scatterings and re-emissions at image bins are recorded (position, w,
// bin) in the peel-off event buffer, one slot range per warp and phase; point-source
// emissions are counted per bin in s_nemit. wt: the warp's counters (shared memory, zero
// at the start; lane 0 or atomics). park: the warp's places. Time budget and counters are
// looked at every `refill_period` steps. Returns false when the time budget ran out.
template <bool kPeel, class Ids, int kS = 0, bool kPath = false, bool kTally = false>
__device__ __forceinline__ bool pool_warp(const DevGrid& g, const DevTables& t, const DevRun& r,
                                          const Kappa* kap, const float* star_cdf,
                                          unsigned long long* sed, unsigned long long n_end,
                                          Ids& ids, LaneTally& tl, unsigned* wt, uint4* park,
                                          unsigned long long t0, const DevPeel* pe = nullptr,
                                          unsigned long long* s_nemit = nullptr,
                                          const float* kext = nullptr,
                                          const float* kabs = nullptr) {
  const int B = g.B;
  const int lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  Pkg<float> k;
  k.id = 0;
  k.dirs = 0;
  bool walking = false;
  bool pending = false;  // reached an interaction point
  // a lane that left the domain is put into the spectrum with the next ones to become
  // idle: until then tau = -1
  k.tau = 0.f;
  // kPath: the path walk (densities from the density array, kI = -kS for the
  // interaction); otherwise the linked walk
  using CellT = typename std::conditional<kPath, PathCell, Cell>::type;
  constexpr int kI = kPath ? -kS : kS;
  constexpr bool kPark = !kTally;
  constexpr int kSteps = kTally ? kTallySteps : kWalkSteps;
  CellT cell{};
  cell.sz = 1.f;
  const int K = r.refill_period > 0 ? min(r.refill_period, 1 << 24) : 32;
  const int n_lanes = r.interaction_batch > 0 ? r.interaction_batch : 8;
  const int batch = kPark ? (n_lanes + 1) / 2 : n_lanes;
  // parked: waiting for their interaction (places 0 ..), ready to walk (the last ones down)
  int n_wait = 0, n_ready = 0;
  bool dry = false;  // no packages left to draw

  // packages that left the domain since into the spectrum
  auto book = [&]() {
    if (k.tau < 0.f) {
      k.tau = 0.f;
      const int db = dir_bin(true_component(k, k.d[2], 2), g.n_dir);
      atomicAdd(&sed[db * B + k.bin], 1ull);
      if (k.event == 0) atomicAdd(&sed[(g.n_dir + db) * B + k.bin], 1ull);
    }
  };
  // new packages for the lanes `dead`
  auto fill = [&](unsigned dead) {
    const bool mine = (dead >> lane) & 1u;
    const unsigned long long j =
        ids.take(__popc(dead), __popc(dead & lt_mask), lane, __ffs(dead) - 1);
    const unsigned fresh = __ballot_sync(kFull, mine && j < n_end);
    dry = fresh != dead;
    if (lane == 0) wt[kCEmitted] += __popc(fresh);
    if (mine && j < n_end) {
      emit<float>(k, r.first_id + j, r, star_cdf, B);
      if constexpr (kPeel) {
        if (r.source_kind != 1) atomicAdd(&s_nemit[k.bin], 1ull);
      }
      int rc;
      if constexpr (kPath)
        rc = enter_path(k, g, cell, tl.levels);
      else
        rc = enter(k, g, cell, tl.levels);
      if (rc == 0) {
        walking = true;
        if constexpr (kPath) cell.kx = path_ext<kS>(g, cell.slot, k.bin, kext);
      } else if (rc == 1) {  // source outside the grid, moving away
        atomicAdd(&wt[kCEscaped], 1u);
        const int db = dir_bin(k.d[2], g.n_dir);
        atomicAdd(&sed[db * B + k.bin], 1ull);
        atomicAdd(&sed[(g.n_dir + db) * B + k.bin], 1ull);
      } else {
        atomicAdd(&wt[kCErrors], 1u);
        atomicOr(r.status, kStatusTree);
      }
    }
  };

  for (;;) {
    if constexpr (!kPark) {
      book();
      const unsigned dead = __ballot_sync(kFull, !walking && !pending);
      if (dead && !dry) fill(dead);
      if (dry && !__any_sync(kFull, walking || pending)) return true;
    }
    if (__any_sync(kFull, tl.crossings >= kTallyFlushAt || tl.levels >= kTallyFlushAt ||
                              wt[lane & (kTallyWords - 1)] >= kTallyFlushAt))
      flush_warp(tl, wt, r.counters);
    bool stop = false;
    if (lane == 0) stop = global_ns() - t0 > r.budget_ns;
    stop = __shfl_sync(kFull, stop, 0);
    if (stop) {
      book();  // what has escaped so far is counted as escaped
      if (lane == 0) atomicOr(r.status, kStatusTimeout);
      return false;
    }
    if constexpr (!kPark) {  // all packages just drawn left the domain at once: draw again
      if (!__any_sync(kFull, walking || pending)) continue;
    }
    for (int step = 0; step < K; ++step) {
      if (walking) {
        int a = kCrossed;
#pragma unroll 2
        for (int u = 0; u < kSteps; ++u) {
          if constexpr (kPath)
            a = advance_path<kS>(k, cell, g, kext, tl.levels);
          else
            a = advance_linked<false, kS, kTally>(k, cell, g, kap, kext, tl.levels, nullptr,
                                                  r.pathabs, kabs);
          if (a != kCrossed) break;
          ++tl.crossings;
        }
        if (a != kCrossed) {
          walking = false;
          if (a == kEscaped) {
            ++tl.crossings;  // the boundary face it left through
            atomicAdd(&wt[kCEscaped], 1u);
            k.tau = -1.f;
          } else if (a == kError) {
            atomicAdd(&wt[kCErrors], 1u);
            k.tau = 0.f;
            atomicOr(r.status, kStatusTree);
          } else {
            pending = true;  // the optical depth runs out inside the cell
          }
        }
      }
      const unsigned wm = __ballot_sync(kFull, walking);
      if constexpr (!kPark) {
        const int np = __popc(__ballot_sync(kFull, pending));
        if (np == 0 || (np < batch && wm)) continue;
      } else {
        if (__popc(wm) > 32 - batch && wm) continue;
        book();
        const unsigned pm = __ballot_sync(kFull, pending);
        const int np = __popc(pm);
        bool act = n_wait + np >= kPlaces;
        if (!act && dry && n_ready == 0) {
          if (wm == 0u && n_wait + np == 0) return true;
          act = wm == 0u || n_wait + np >= batch;
          if (!act) continue;
        }
        bool load = false, store = false, refill = false;
        int src = 0, dst = 0;
        if (act) {
          const unsigned dm = ~(wm | pm);
          const int nd = __popc(dm), n = min(n_wait, 32 - np);
          const int rank = walking ? nd + __popc(wm & lt_mask) : __popc(dm & lt_mask);
          load = !pending && rank < n;
          store = load && walking;
          src = n_wait - 1 - rank;
          dst = kPlaces - 1 - n_ready - (rank - nd);
          n_wait -= n;
          n_ready += max(n - nd, 0);
        } else if (n_ready > 0) {
          const int rank = __popc(~wm & lt_mask), n = min(n_ready, 32 - __popc(wm));
          load = !walking && rank < n;
          store = load && pending;
          const unsigned sm = __ballot_sync(kFull, store);
          src = kPlaces - n_ready + rank;
          dst = n_wait + __popc(sm & lt_mask);
          n_ready -= n;
          n_wait += __popc(sm);
        } else {
          store = pending;
          dst = n_wait + __popc(pm & lt_mask);
          n_wait += np;
          refill = true;
        }
        if (__any_sync(kFull, load || store)) {
          park_exchange<kPath>(park, k, cell, load, src, store, dst);
          if (load) {
            walking = !act;
            pending = act;
            set_inverse(k);
          } else if (store) {
            pending = false;
          }
        }
        if (refill) fill(~wm);
        if (!act) continue;
      }
      // interactions
      int sp = -1;
      uint4 w1 = make_uint4(0, 0, 0, 0);
      bool absorbing = false;
      bool scattered = false;
      float wv = kInv4Pi;  // peel-off weight per steradian of this lane's event
      int leaf = 0, row = 0;  // the cell's leaf id; its density row (leaf or slot)
      if (pending) {
        pending = false;
        walking = true;
        float kx;
        if constexpr (kPath)
          kx = cell.kx;
        else
          kx = leaf_ext<kS, kTally>(g, cell.leaf, leaf_rho<kS>(g, cell.leaf), k.bin, kap, kext);
        to_point(k, cell, kx);
        if constexpr (kPath) {
          leaf = path_leaf(g, cell.slot);
          row = kI < 0 ? cell.slot : leaf;  // slot rows for 2 or 4 species
        } else {
          leaf = cell.leaf;
          row = leaf;
        }
        if (++k.event > r.max_events) {
          atomicAdd(&wt[kCCapped], 1u);
          walking = false;
          k.tau = 0.f;
        } else if (leaf < 0) {
          atomicAdd(&wt[kCErrors], 1u);
          atomicOr(r.status, kStatusTree);
          walking = false;
          k.tau = 0.f;
        } else {
          const unsigned was = mirrored(k);
          restore_direction(k);
          sp = interact<float, kI>(k, g, kap, row, r, w1, kPeel ? pe->o : nullptr,
                                   kPeel ? &wv : nullptr);
          orient<kPath>(k, cell, was);
          if (sp < 0) {
            scattered = true;
          } else {
            absorbing = true;
          }
        }
      }
      const unsigned am = __ballot_sync(kFull, absorbing);
      const unsigned sm = __ballot_sync(kFull, scattered);
      if (lane == 0) {
        wt[kCAbsorptions] += __popc(am);
        wt[kCScatters] += __popc(sm);
      }
      if (absorbing) {
        unsigned long long key = ((unsigned long long)sp << 48) | (unsigned long long)leaf;
        unsigned peers = __match_any_sync(am, key);
        int leader = __ffs(peers) - 1;
        unsigned long long old = 0;
        if (lane == leader)
          old = atomicAdd(&r.count[(size_t)sp * g.n_leaves + leaf],
                          (unsigned long long)__popc(peers));
        old = __shfl_sync(peers, old, leader);
        if (t.pah_of[sp] >= 0)
          pah_absorb<float>(k, g, t, r, t.pah_of[sp], leaf, w1);
        else {
          unsigned clamped = 0;
          reemit<float, kI>(k, g, t, r, sp, leaf, row, cell.level(), old + __popc(peers & lt_mask),
                            w1, clamped);
          if (clamped) atomicAdd(&wt[kCClamped], 1u);
        }
        if constexpr (kPath) cell.kx = path_ext<kS>(g, cell.slot, k.bin, kext);
      }
      if constexpr (kPeel) {
        // the event's share toward the observer, at the bin it leaves with
        const bool ev = (scattered || absorbing) && __ldg(&pe->plane_of_bin[k.bin]) >= 0;
        const unsigned em = __ballot_sync(kFull, ev);
        if (em) {
          const int leader = __ffs(em) - 1;
          unsigned long long base = 0;
          if (lane == leader) base = atomicAdd(pe->n_ev, (unsigned long long)__popc(em));
          base = __shfl_sync(kFull, base, leader);
          if (ev) {
            const unsigned long long slot = base + __popc(em & lt_mask);
            if (slot < pe->capacity) {
              pe->ev[slot] = make_float4(true_component(k, k.p[0], 0), true_component(k, k.p[1], 1),
                                         true_component(k, k.p[2], 2), wv);
              pe->ev_bin[slot] = k.bin;
            }
          }
          if (lane == leader) wt[kCPeelEvents] += __popc(em);
        }
      }
    }
  }
}

// Shared-memory words (floats) of the extinction opacities [B][S], rounded up to 16 bytes, and
// the opacity records staged there too. A crossing needs the extinctions alone: with the
// records of a generic walk's species in every block, beside the places, nothing was left of L1
// (1e6 packages through 1.1e5 cells, ms, records and extinctions in shared memory: five
// species, 400 bins 1.78 and 1.01; six 1.92 and 1.28; eight, 200 bins 2.74 and 2.33; five, 100
// bins 0.98 and 0.95). Records are read at interactions, from L1, but for two species (4.11 ms
// in shared memory against 4.17 for the disk of 2.4e6 cells) and for the generic walk with the
// path-length tally, which reads them at every crossing and has no places.
template <int kS, bool kTally>
__host__ __device__ __forceinline__ int kext_words(const DevGrid& g) {
  return kS == 0 && kTally ? 0 : (g.B * (kS > 0 ? kS : g.S) + 3) / 4 * 4;
}

template <int kS, bool kTally>
__host__ __device__ __forceinline__ int kap_records(const DevGrid& g) {
  return kS == 2 || (kS == 0 && kTally) ? g.B * g.S : 0;
}

// ---------------------------------------------------------------- pool kernel
// Shared memory of a warp: its places and its counters.
template <bool kPath, bool kTally>
__host__ __device__ constexpr int pool_warp_bytes() {
  return (kTally ? 0 : park_bytes<kPath>()) + 4 * kTallyWords;
}

// Persistent packet pool over one model: all warps draw package indices from one
// global counter; the opacity table, the stellar CDF and (where that costs no resident
// block: launch_pool_variant) the escaped-spectrum histogram live in shared memory.
template <int kMinBlocks, bool kPeel, int kS = 0, bool kPath = false, bool kTally = false>
__global__ void __launch_bounds__(256, kMinBlocks)
    k_transport_pool(DevGrid g, DevTables t, DevRun r, const __grid_constant__ DevPeel pe) {
  extern __shared__ __align__(16) unsigned char smem[];
  // the warps' places and counters (as many as the block has warps: eight for blocks of any
  // size left the smaller ones a few KB of L1; 1e6 packages through 1.1e5 cells, blocks of 128:
  // five species 1.77 against 1.13 ms), then the launch's tables
  constexpr int kWarpBytes = pool_warp_bytes<kPath, kTally>();
  unsigned char* mine = smem + (threadIdx.x >> 5) * kWarpBytes;
  unsigned* wt = reinterpret_cast<unsigned*>(mine + kWarpBytes - 4 * kTallyWords);
  uint4* park = reinterpret_cast<uint4*>(mine);
  if ((threadIdx.x & 31) < kTallyWords) wt[threadIdx.x & 31] = 0u;
  unsigned long long* smem_u64 =
      reinterpret_cast<unsigned long long*>(smem + (blockDim.x >> 5) * kWarpBytes);
  const int S = g.S, B = g.B;
  const int n_sed = 2 * g.n_dir * B;
  const bool sed_local = r.sed_in_smem != 0;
  // the extinction opacities [B][S] first (with the path-length tally of 2 or 4 species the
  // absorption opacities after them), for 2 or 4 one vector per bin (a multiple of 16 bytes)
  float* s_kext = reinterpret_cast<float*>(smem_u64);
  const int n_kext = kext_words<kS, kTally>(g);
  float* s_kabs = s_kext + n_kext;
  unsigned long long* s_u64 = smem_u64 + (kTally ? 2 : 1) * n_kext / 2;
  unsigned long long* s_sed = sed_local ? s_u64 : r.sed;   // [2][n_dir][B]
  Kappa* s_kap = reinterpret_cast<Kappa*>(s_u64 + (sed_local ? n_sed : 0));  // [B][S]
  const int n_kap = kap_records<kS, kTally>(g);
  float* s_cdf = reinterpret_cast<float*>(s_kap + n_kap);     // [B]
  if (sed_local)
    for (int i = threadIdx.x; i < n_sed; i += blockDim.x) s_sed[i] = 0ull;
  if (n_kap)
    for (int i = threadIdx.x; i < n_kap; i += blockDim.x) s_kap[i] = t.kap[i];
  if (n_kext)
    for (int i = threadIdx.x; i < B * S; i += blockDim.x) {
      s_kext[i] = t.kext[i];
      if (kTally) s_kabs[i] = t.kap[i].kabs;
    }
  for (int i = threadIdx.x; i < B; i += blockDim.x) s_cdf[i] = t.star_cdf[i];
  // peel-off: the block's point-source emission counts per bin
  unsigned long long* s_nemit = nullptr;
  if constexpr (kPeel) {
    const uintptr_t a = (reinterpret_cast<uintptr_t>(s_cdf + B) + 15) & ~(uintptr_t)15;
    s_nemit = reinterpret_cast<unsigned long long*>(a);
    for (int i = threadIdx.x; i < B; i += blockDim.x) s_nemit[i] = 0ull;
  }
  __syncthreads();
  LaneTally tl = {};
  GlobalIds ids{r.next};
  pool_warp<kPeel, GlobalIds, kS, kPath, kTally>(g, t, r, kS == 2 || (kS == 0 && kTally) ? s_kap : t.kap, s_cdf, s_sed,
                                                 r.n_packages, ids, tl, wt, park, global_ns(), &pe,
                                                 s_nemit, s_kext, s_kabs);
  flush_warp(tl, wt, r.counters);
  if (sed_local || kPeel) __syncthreads();
  if (sed_local) {
    for (int i = threadIdx.x; i < n_sed; i += blockDim.x)
      if (s_sed[i]) atomicAdd(&r.sed[i], s_sed[i]);
  }
  if constexpr (kPeel) {
    for (int i = threadIdx.x; i < B; i += blockDim.x)
      if (s_nemit[i]) atomicAdd(&pe.n_emit[i], s_nemit[i]);
  }
}

// ---------------------------------------------------------------- batch kernel
// Many models in one persistent launch. A warp picks a model, stages its descriptor in
// shared memory and runs the pool loop on it, drawing packages from the model's counter
// until that is exhausted and its own lanes have run dry; then it picks the next. The
// pick is weighted by the packages each model has left (pick_model): the first one stratified over
// the warps (so that neighbouring warps share a model's rows in L1), later ones at
// random. A warp's lanes therefore run dry once per model it works on. (Fixed chunks of
// 4096 packages, a warp's lanes drained at the end of each, left three quarters of the
// warps without work for a batch of 24 models and 6.5e6 packages -- 1600 chunks for 4864
// warps -- and took 28.7 ms against 8.0 for this, and 4.8 with the walk as it is now.) Tables
// in global memory / L2, spectrum by global atomics; counters are flushed to the model when
// the warp leaves it.
//
// Up to kPickWindow models are weighed together by what each has left. Of more, one is drawn by
// the plan (its packages at the start) and taken if it has any left, else the window of models
// from it on is weighed, and so on round the batch: a pick's cost does not grow with the batch
// until its end, and then only while some model has packages. (Weighing all models at every pick, with their descriptors read for it, 4000 and
// 8000 models of 50 packages took 565 and 1427 us beside 87 and 148 for chunks of one model; now
// 96 and 182.)
constexpr int kPickWindow = 256;

__device__ __forceinline__ int pick_model(const BatchQueue& q, unsigned warp_id, unsigned n_warps,
                                          unsigned pick) {
  const int lane = threadIdx.x & 31;
  auto remaining = [&](int m) {
    const unsigned long long all = q.plan[m];
    const unsigned long long out =
        *reinterpret_cast<const volatile unsigned long long*>(&q.next[m]);
    return out < all ? all - out : 0ull;
  };
  // a point as a 64-bit fraction: the warp's place, or a hash
  unsigned long long frac = (((unsigned long long)warp_id << 1 | 1) << 31) / n_warps << 32;
  if (pick > 0) {
    frac = ((unsigned long long)warp_id << 32 | pick) * 0x9E3779B97F4A7C15ull;
    frac ^= frac >> 29;
    frac *= 0xBF58476D1CE4E5B9ull;
  }
  int first = 0;
  if (q.n > kPickWindow) {
    const unsigned long long point = __umul64hi(frac, q.before[q.n]);
    int hi = q.n;  // before[first] <= point < before[hi]
    while (hi - first > 1) {
      const int mid = (first + hi) >> 1;
      if (q.before[mid] <= point) first = mid; else hi = mid;
    }
    if (__shfl_sync(kFull, remaining(first), 0) > 0) return first;
    const unsigned long long done =
        *reinterpret_cast<const volatile unsigned long long*>(&q.next[q.n]);
    if (__shfl_sync(kFull, done, 0) >= (unsigned long long)q.n_live) return -1;
    frac = (frac ^ frac >> 31) * 0x94D049BB133111EBull;
  }
  for (int off = 0; off < q.n; off += kPickWindow) {
    constexpr int kEach = kPickWindow / 32;
    unsigned long long r[kEach], sum = 0;
#pragma unroll
    for (int j = 0; j < kEach; ++j) {
      const int i = off + 32 * j + lane, m = first + i;
      r[j] = i < q.n ? remaining(m < q.n ? m : m - q.n) : 0ull;
      sum += r[j];
    }
    unsigned long long c = sum;  // inclusive sum over the lanes
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long u = __shfl_up_sync(kFull, c, o);
      if (lane >= o) c += u;
    }
    const unsigned long long tot = __shfl_sync(kFull, c, 31);
    if (tot == 0) continue;
    const unsigned long long point = __umul64hi(frac, tot);
    const int src = __ffs(__ballot_sync(kFull, c > point)) - 1;
    unsigned long long p = point - (c - sum);  // within the lane src
    int at = off + lane;
#pragma unroll
    for (int j = 0; j + 1 < kEach; ++j)
      if (at == off + 32 * j + lane && p >= r[j]) {
        p -= r[j];
        at += 32;
      }
    const int m = first + __shfl_sync(kFull, at, src);
    return m < q.n ? m : m - q.n;
  }
  return -1;
}

// Two species: held to 64 registers (46 bytes of spills) for four blocks per SM; when this
// was decided 8.0 ms against 8.7 with three blocks of 74 registers, and 180 bytes of spills in
// the generic form.
template <int kS, bool kTally>
__global__ void __launch_bounds__(256, kS == 2 ? 4 : 3) k_transport_batch(const ModelDesc* models,
                                                         BatchQueue q, int chunk) {
  __shared__ ModelDesc sdesc[8];
  __shared__ unsigned s_tally[8 * kTallyWords];
  constexpr int kParkBytes = kTally ? 16 : park_bytes<false>();
  __shared__ __align__(16) unsigned char s_park[8 * kParkBytes];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint4* park = reinterpret_cast<uint4*>(s_park + warp * kParkBytes);
  unsigned* wt = s_tally + warp * kTallyWords;
  if (lane < kTallyWords) wt[lane] = 0u;
  const unsigned per_block = blockDim.x >> 5;
  const unsigned long long t0 = global_ns();
  for (unsigned pick = 0;; ++pick) {
    const int m = pick_model(q, blockIdx.x * per_block + warp, gridDim.x * per_block, pick);
    if (m < 0) break;
    const int* src = reinterpret_cast<const int*>(&models[m]);
    int* dst = reinterpret_cast<int*>(&sdesc[warp]);
    for (int i = lane; i < (int)(sizeof(ModelDesc) / sizeof(int)); i += 32) dst[i] = src[i];
    __syncwarp();
    const ModelDesc& md = sdesc[warp];
    LaneTally tl = {};
    ModelIds ids{q.next + m, 0ull, md.r.n_packages, 0, chunk};
    const bool in_time =
        pool_warp<false, ModelIds, kS, false, kTally>(md.g, md.t, md.r, md.t.kap, md.t.star_cdf, md.r.sed,
                                        md.r.n_packages, ids, tl, wt, park, t0, nullptr, nullptr,
                                        md.t.kext);
    flush_warp(tl, wt, md.r.counters);
    __syncwarp();
    if (in_time && lane == 0 && !(atomicOr(&q.next[m], kExhausted) & kExhausted))
      atomicAdd(&q.next[q.n], 1ull);
    if (!in_time) {
      // the budget is the launch's: what is left of any model stays undone, and its status
      // says so, also where no warp was on it (models with few packages wait for the large)
      for (int j = lane; j < q.n; j += 32)
        if (*reinterpret_cast<const volatile unsigned long long*>(&q.next[j]) < q.plan[j])
          atomicOr(models[j].r.status, kStatusTimeout);
      break;
    }
  }
}

// ---------------------------------------------------------------- replay
// Frozen mode only: counts do not steer the path, so each listed package is
// followed alone and its history recorded.
// ev (optional): the package's events, at most ev_cap of them at ev + i ev_cap;
// ev_n[i] receives how many the history has.
__device__ __forceinline__ void trace_event(TraceEvent* ev, long long cap, long long& n,
                                            int kind, int species, int leaf, int bin,
                                            const float p[3]) {
  if (ev && n < cap) {
    TraceEvent e;
    e.kind = kind;
    e.species = species;
    e.leaf = leaf;
    e.bin = bin;
    e.pos[0] = p[0];
    e.pos[1] = p[1];
    e.pos[2] = p[2];
    e.pad = 0;
    ev[n] = e;
  }
  ++n;
}

__global__ void k_trace(DevGrid g, DevTables t, DevRun r, const unsigned long long* ids,
                        long long n, long long* out, TraceEvent* ev, long long ev_cap,
                        long long* ev_n) {
  long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  TraceEvent* my_ev = ev ? ev + i * ev_cap : nullptr;
  long long n_ev = 0;
  Tally tl = {};
  Pkg<float> k;
  emit<float>(k, ids[i], r, t.star_cdf, g.B);
  trace_event(my_ev, ev_cap, n_ev, 0, -1, -1, k.bin, k.p);
  long long rec[9] = {0, 0, 0, 0, 0, 0, 0, 0, -1};
  const unsigned long long t0 = global_ns();
  unsigned steps = 0;
  Cell c{0, {0.f, 0.f, 0.f}, 1.f};
  k.dirs = 0;
  int rc = enter(k, g, c, tl.levels);
  auto at = [&](int a) { return true_component(k, k.p[a], a); };
  if (rc == 1) rec[4] = 1;
  if (rc < 0) atomicOr(r.status, kStatusTree);
  while (rc == 0) {
    if ((++steps & 1023u) == 0 && global_ns() - t0 > r.budget_ns) {
      atomicOr(r.status, kStatusTimeout);
      break;
    }
    const int lf = c.leaf;
    const int a = advance_linked(k, c, g, t.kap, t.kext, tl.levels);
    rec[8] = lf;
    if (a == kCrossed) { ++rec[3]; continue; }
    if (a == kEscaped) {
      ++rec[3];
      rec[4] = 1;
      const float pe[3] = {at(0), at(1), at(2)};
      trace_event(my_ev, ev_cap, n_ev, 3, -1, lf, k.bin, pe);
      break;
    }
    if (a == kError) { atomicOr(r.status, kStatusTree); break; }
    to_point(k, c, leaf_ext<0>(g, c.leaf, float4{}, k.bin, t.kap, t.kext));
    const float pi[3] = {at(0), at(1), at(2)};
    if (++k.event > r.max_events) {
      rec[5] = 1;
      trace_event(my_ev, ev_cap, n_ev, 4, -1, c.leaf, k.bin, pi);
      break;
    }
    uint4 w1;
    const unsigned was = mirrored(k);
    restore_direction(k);
    int s = interact<float>(k, g, t.kap, c.leaf, r, w1);
    orient<false>(k, c, was);
    if (s < 0) {
      ++rec[2];
      trace_event(my_ev, ev_cap, n_ev, 1, -1, c.leaf, k.bin, pi);
      continue;
    }
    if (t.pah_of[s] >= 0) {
      pah_bin(k, g, t, t.pah_of[s], c.leaf, w1);  // replay does not tally
    } else {
      reemit<float>(k, g, t, r, s, c.leaf, c.leaf, c.level(), 0ull, w1, tl.clamped);
    }
    trace_event(my_ev, ev_cap, n_ev, 2, s, c.leaf, k.bin, pi);
    ++rec[1];
  }
  if (ev_n) ev_n[i] = n_ev;
  rec[0] = k.event;
  rec[6] = k.bin;
  rec[7] = dir_bin(true_component(k, k.d[2], 2), g.n_dir);
  for (int j = 0; j < 9; ++j) out[i * 9 + j] = rec[j];
}

// Rows by tree slot (the path walk's grid): slot i < n^3 is base cell i, slot
// n^3 + 8 b + o the child o of block b. A leaf's row holds its densities (a -0 made
// +0: the densities are non-negative); a refined slot's row holds the code -(block +
// 1) of its block in the first word, zeros after it.
__global__ void k_build_rho_slot(DevGrid g, long long n_slots, float* out) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n_slots) return;
  const long long nb = g.n_base3;
  const int node = i < nb ? g.base[i] : g.child[i - nb];
  const bool leaf = node >= 0 && node < g.n_leaves;
  for (int s = 0; s < g.S; ++s)
    out[i * g.S + s] = leaf ? fabsf(g.rho[(long long)node * g.S + s])
                            : (s == 0 && node < 0 ? __int_as_float(node) : 0.f);
}

// Face links: for each leaf and face, the neighbour across it at the leaf's level
// (descending from the base cube with integer coordinates).
__global__ void k_build_links(DevGrid g, const int32_t* ijk, int32_t* links) {
  long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (idx >= g.n_leaves * 6) return;
  const long long leaf = idx / 6;
  const int f = (int)(idx % 6), a = f >> 1;
  const int lev = g.level[leaf];
  int J[3] = {ijk[leaf * 3], ijk[leaf * 3 + 1], ijk[leaf * 3 + 2]};
  J[a] += (f & 1) ? 1 : -1;
  const long long nl = (long long)g.n_base << lev;
  int32_t link;
  if (J[a] < 0 || J[a] >= nl) {
    link = kLinkEscape;
  } else {
    const int n = g.n_base;
    int node = g.base[(J[0] >> lev) + n * ((J[1] >> lev) + n * (J[2] >> lev))];
    int l = 0;
    while (node < 0 && l < lev) {
      const long long blk = -(long long)node - 1;
      ++l;
      const int sh = lev - l;
      const int oct = ((J[0] >> sh) & 1) | (((J[1] >> sh) & 1) << 1) | (((J[2] >> sh) & 1) << 2);
      node = g.child[blk * 8 + oct];
    }
    link = node >= 0 ? (node | ((lev - l) << 28)) : node;
  }
  int32_t* rec = links + leaf * kRec;
  rec[f] = link;
  if (f == 0) {
    rec[6] = g.S >= 1 && g.S <= 2 ? __float_as_int(g.rho[leaf * g.S]) : 0;
    rec[7] = g.S == 2 ? __float_as_int(g.rho[leaf * g.S + 1]) : 0;
  }
}

__global__ void k_philox(const unsigned long long* ids, long long n, unsigned event,
                         unsigned block, unsigned long long seed, unsigned* out) {
  long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint4 w = draw(seed, ids[i], event, block);
  out[4 * i] = w.x;
  out[4 * i + 1] = w.y;
  out[4 * i + 2] = w.z;
  out[4 * i + 3] = w.w;
}

}  // namespace

constexpr size_t kSmemBudget = 200 * 1024;
constexpr size_t kSmemBlock = 1024;  // kept by each block beside what it asks for
// shared memory of an SM beyond which the next carve-outs leave L1 a quarter or less of the 256 KB
constexpr size_t kSmemKeep = 164 * 1024;

template <int kS, bool kTally>
static size_t table_smem(const DevGrid& g) {
  return sizeof(Kappa) * kap_records<kS, kTally>(g) +
         sizeof(float) * ((kTally ? 2 : 1) * kext_words<kS, kTally>(g) + g.B);
}

static size_t sed_smem(const DevGrid& g) {
  return sizeof(unsigned long long) * 2 * g.n_dir * g.B;
}

static size_t peel_smem(const DevGrid& g) { return 16 + sizeof(unsigned long long) * g.B; }

template <int kMinBlocks, bool kPeel, int kS = 0, bool kPath = false, bool kTally = false>
static cudaError_t launch_pool_variant(const DevGrid& g, const DevTables& t, const DevRun& r,
                                       const DevPeel& pe, int blocks_per_sm, int threads,
                                       int sms, cudaStream_t s) {
  DevRun rr = r;
  const size_t tables = table_smem<kS, kTally>(g) + (kPeel ? peel_smem(g) : 0);
  const size_t warps = threads / 32 * pool_warp_bytes<kPath, kTally>();
  rr.sed_in_smem = tables + sed_smem(g) <= kSmemBudget ? 1 : 0;
  size_t sm = warps + tables + (rr.sed_in_smem ? sed_smem(g) : 0);
  cudaError_t e;
  const auto kernel = k_transport_pool<kMinBlocks, kPeel, kS, kPath, kTally>;
  if (sm > 48 * 1024) {
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
  }
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, sm);
  if (e != cudaSuccess) return e;
  // The spectrum in shared memory is worth a few per cent, a block per SM or L1 far more: it goes
  // to global memory where, beside the places, it would cost a block that the launch would have,
  // or L1 (asked only where shared memory can be what limits). 5.3e5 cells of two species,
  // 3e6 packages, in shared and in global memory, ms: 200 bins, one direction (four blocks
  // both) 1.28 and 1.30; eight directions of 257 bins (three and four) 1.57 and 1.29, path
  // walk 2.69 and 2.27; of 333 bins (two and four) 2.28 and 1.29, path walk 3.53 and 2.28; of
  // 1024 bins (one and four) 3.61 and 1.58. Four blocks both, 1e6 packages through 1.1e5 cells:
  // three species, 1024 bins 1.45 and 0.81, two species, 600 bins 0.86 and 0.59.
  if (rr.sed_in_smem && (sm + kSmemBlock) * kMinBlocks * 256 > kSmemKeep * threads) {
    int most = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&most, kernel, threads, warps + tables);
    if (e != cudaSuccess) return e;
    const int want = blocks_per_sm > 0 && blocks_per_sm < most ? blocks_per_sm : most;
    if (occ < want || (sm + kSmemBlock) * want > kSmemKeep) {
      rr.sed_in_smem = 0;
      sm = warps + tables;
      occ = most;
    }
  }
  if (occ < 1) occ = 1;
  int bps = blocks_per_sm > 0 ? (blocks_per_sm < occ ? blocks_per_sm : occ) : occ;
  kernel<<<sms * bps, threads, sm, s>>>(g, t, rr, pe);
  return cudaGetLastError();
}

// blocks_per_sm selects the register budget: 5 or 6 resident blocks of 256 threads
// use variants compiled for that occupancy (fewer registers, some spills); other
// values use the 4-block variants, capped at their occupancy: the walks compiled for two
// or four species or the generic one. With peel-off images or the path-length tally the
// 4-block variants are used.
//
// Four is also what they take left to themselves (0): five blocks give the walks of two or
// four species 48 registers, which spill now that packages move between lanes and places,
// and their places take shared memory from L1 (2.4e6 cells, 5e6 packages: 3.40 ms against 3.21).
cudaError_t launch_transport_pool(const DevGrid& g, const DevTables& t, const DevRun& r,
                                  int blocks_per_sm, int threads, cudaStream_t s,
                                  const DevPeel* peel, bool path) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  if (peel && r.pathabs)
    return launch_pool_variant<4, true, 0, false, true>(g, t, r, *peel, blocks_per_sm, threads,
                                                        sms, s);
  if (peel && g.S == 2)
    return launch_pool_variant<4, true, 2>(g, t, r, *peel, blocks_per_sm, threads, sms, s);
  if (peel) return launch_pool_variant<4, true>(g, t, r, *peel, blocks_per_sm, threads, sms, s);
  const DevPeel none{};
  // the path-length tally: the linked walk, at four blocks per SM
  if (r.pathabs) {
    if (g.S == 2)
      return launch_pool_variant<4, false, 2, false, true>(g, t, r, none, blocks_per_sm, threads,
                                                           sms, s);
    if (g.S == 4)
      return launch_pool_variant<4, false, 4, false, true>(g, t, r, none, blocks_per_sm, threads,
                                                           sms, s);
    return launch_pool_variant<4, false, 0, false, true>(g, t, r, none, blocks_per_sm, threads,
                                                         sms, s);
  }
  // the path walk (no face links; grids of at most kPathLevels levels)
  if (path && g.max_level <= kPathLevels) {
    if (g.S == 4)
      return launch_pool_variant<4, false, 4, true>(g, t, r, none, blocks_per_sm, threads, sms, s);
    if (g.S == 2)
      return launch_pool_variant<4, false, 2, true>(g, t, r, none, blocks_per_sm, threads, sms, s);
    return launch_pool_variant<4, false, 0, true>(g, t, r, none, blocks_per_sm, threads, sms, s);
  }
  if (threads == 256 && blocks_per_sm == 6)
    return launch_pool_variant<6, false>(g, t, r, none, blocks_per_sm, threads, sms, s);
  if (threads == 256 && blocks_per_sm == 5)
    return launch_pool_variant<5, false>(g, t, r, none, blocks_per_sm, threads, sms, s);
  if (g.S == 2)
    return launch_pool_variant<4, false, 2>(g, t, r, none, blocks_per_sm, threads, sms, s);
  if (g.S == 4)
    return launch_pool_variant<4, false, 4>(g, t, r, none, blocks_per_sm, threads, sms, s);
  return launch_pool_variant<4, false>(g, t, r, none, blocks_per_sm, threads, sms, s);
}

cudaError_t launch_peel_source(const DevGrid& g, const DevTables& t, const DevRun& r,
                               const DevPeel& peel, cudaStream_t s) {
  k_peel_source<<<(g.B + 127) / 128, 128, 0, s>>>(g, t, r, peel);
  return cudaGetLastError();
}

cudaError_t launch_peel_trace(const DevGrid& g, const DevTables& t, const DevRun& r,
                              const DevPeel& peel, cudaStream_t s) {
  int dev = 0, sms = 0, occ = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_peel_trace, 256, 0);
  if (e != cudaSuccess) return e;
  k_peel_trace<<<sms * (occ > 0 ? occ : 1), 256, 0, s>>>(g, t, r, peel);
  return cudaGetLastError();
}

cudaError_t launch_image_out(const double* image, long long n, double scale, double* out,
                             cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_image_out<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(image, n, scale, out);
  return cudaGetLastError();
}

cudaError_t launch_image_profile(const double* image, int nx, int ny, int plane_a,
                                 int plane_b, int half_rows, double scale, double* out,
                                 cudaStream_t s) {
  k_image_profile<<<(nx + 127) / 128, 128, 0, s>>>(image, nx, ny, plane_a, plane_b, half_rows,
                                                    scale, out);
  return cudaGetLastError();
}

cudaError_t launch_transport_plain(const DevGrid& g, const DevTables& t, const DevRun& r,
                                   bool fp64, int threads, cudaStream_t s) {
  unsigned long long nb = (r.n_packages + threads - 1) / threads;
  if (nb == 0) return cudaSuccess;
  if (nb > 0x7fffffffull) return cudaErrorInvalidValue;
  const auto kernel = r.pathabs ? (fp64 ? k_transport_plain<double, true>
                                        : k_transport_plain<float, true>)
                                : (fp64 ? k_transport_plain<double, false>
                                        : k_transport_plain<float, false>);
  kernel<<<(unsigned)nb, threads, 0, s>>>(g, t, r);
  return cudaGetLastError();
}

template <int kS, bool kTally>
static cudaError_t launch_batch_variant(const ModelDesc* models, const BatchQueue& q, int chunk,
                                        int blocks_per_sm, int threads, cudaStream_t s) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_transport_batch<kS, kTally>, threads, 0);
  if (e != cudaSuccess) return e;
  if (occ < 1) occ = 1;
  int bps = blocks_per_sm > 0 && blocks_per_sm < occ ? blocks_per_sm : occ;
  k_transport_batch<kS, kTally><<<sms * bps, threads, 0, s>>>(models, q, chunk);
  return cudaGetLastError();
}

cudaError_t launch_transport_batch(const ModelDesc* models, const BatchQueue& q, int chunk,
                                   int blocks_per_sm, int s_fixed, bool tally, int threads,
                                   cudaStream_t s) {
  if (threads <= 0) threads = 256;
  if (threads % 32 != 0 || threads > 256) return cudaErrorInvalidValue;
  if (tally)
    return launch_batch_variant<0, true>(models, q, chunk, blocks_per_sm, threads, s);
  if (s_fixed == 2)
    return launch_batch_variant<2, false>(models, q, chunk, blocks_per_sm, threads, s);
  return launch_batch_variant<0, false>(models, q, chunk, blocks_per_sm, threads, s);
}

cudaError_t launch_trace(const DevGrid& g, const DevTables& t, const DevRun& r,
                         const unsigned long long* ids, long long n, long long* out,
                         cudaStream_t s, TraceEvent* ev, long long ev_cap, long long* ev_n) {
  if (n <= 0) return cudaSuccess;
  k_trace<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(g, t, r, ids, n, out, ev, ev_cap,
                                                      ev_n);
  return cudaGetLastError();
}

cudaError_t launch_build_links(const DevGrid& g, const int32_t* leaf_ijk, int32_t* links,
                               cudaStream_t s) {
  long long n = g.n_leaves * 6;
  k_build_links<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(g, leaf_ijk, links);
  return cudaGetLastError();
}

cudaError_t launch_build_rho_slot(const DevGrid& g, float* rho_slot, cudaStream_t s) {
  const long long n = (long long)g.n_base3 + 8 * g.n_blocks;
  k_build_rho_slot<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(g, n, rho_slot);
  return cudaGetLastError();
}

cudaError_t launch_philox(const unsigned long long* ids, long long n, unsigned event,
                          unsigned block, unsigned long long seed, unsigned* out,
                          cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_philox<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(ids, n, event, block, seed, out);
  return cudaGetLastError();
}

}  // namespace rt
