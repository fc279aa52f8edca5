// rt_tables.cu -- FP64 table builders, frozen-temperature energies and the
// per-cell temperature update of librt_gb300 (Planck integrals: rt_planck.cuh).

#include "rt_internal.h"
#include "rt_planck.cuh"

#include <math.h>

namespace rt {
namespace {

using namespace planck;

// Inclusive sum over the warp's lanes.
__device__ __forceinline__ double scan_add(double v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double u = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += u;
  }
  return v;
}

// Inclusive maximum over the warp's lanes.
__device__ __forceinline__ float scan_max(float v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float u = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v = fmaxf(v, u);
  }
  return v;
}

// One warp: the normalised cumulative of v(b) >= 0, b = 0 .. B-1, into out (1 where the
// sum is not positive; the last entry exactly 1). The sum runs in FP64 by a scan of 32
// bins at a time; a running maximum after rounding keeps the entries in order where the
// scan's different groupings differ in the last bit. Returns the sum.
template <typename F, typename G>
__device__ __forceinline__ double cumulative_warp(int B, F v, G out) {
  const int lane = threadIdx.x & 31;
  double tot = 0.0;
  for (int b = lane; b < B; b += 32) tot += v(b);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
  double carry = 0.0;
  float top = 0.0f;
  for (int b0 = 0; b0 < B; b0 += 32) {
    const int b = b0 + lane;
    const double c = scan_add(b < B ? v(b) : 0.0);
    const float m = fmaxf(top, scan_max(tot > 0.0 ? (float)((carry + c) / tot) : 1.0f));
    if (b < B) out(b, b == B - 1 ? 1.0f : m);
    carry += __shfl_sync(0xffffffffu, c, 31);
    top = __shfl_sync(0xffffffffu, m, 31);
  }
  return tot;
}

// Opacity records of a bin.
__device__ __forceinline__ void opacities(const TableBuild& tb, int b) {
  for (int s = 0; s < tb.S; ++s) {
    size_t j = (size_t)s * tb.B + b;
    Kappa k;
    k.kabs = (float)tb.kabs[j];
    k.ksca = (float)tb.ksca[j];
    k.kext = (float)(tb.kabs[j] + tb.ksca[j]);
    k.g = (float)tb.ghg[j];
    tb.kap[(size_t)b * tb.S + s] = k;
    tb.kext[(size_t)b * tb.S + s] = k.kext;
  }
}

// Stellar CDF and the in-range fraction of the blackbody: the bin edges in parallel
// (one block), the cumulative by one warp. (The integrals bin by bin with the division
// of every entry in one thread took 0.46 ms for 100 bins; this takes 0.03 ms.)
__device__ __forceinline__ void star_spectrum(const TableBuild& tb, double* edge) {
  const int B = tb.B;
  const double a = kH / (kK * tb.T_star), pref = planck_factor(tb.T_star);
  for (int b = threadIdx.x; b <= B; b += blockDim.x) edge[b] = planck_edge(a * tb.nu[b]);
  __syncthreads();
  if (threadIdx.x >= 32) return;
  const double tot = cumulative_warp(
      B,
      [&](int b) {
        return pref * planck_between(a * tb.nu[b], edge[b], a * tb.nu[b + 1], edge[b + 1]);
      },
      [&](int b, float c) { tb.star_cdf[b] = c; });
  if (threadIdx.x == 0) {
    // sigma = 2 pi^5 k^4 / (15 c^2 h^3)
    double sigma = 2.0 * pow(kPi, 5.0) * pow(kK, 4.0) / (15.0 * kC * kC * pow(kH, 3.0));
    double T4 = pow(tb.T_star, 4.0);
    tb.star_frac[0] = kPi * tot / (sigma * T4);
  }
}

// One block per table row: the row's bin edges once each (FP64 is the cost: see
// rt_planck.cuh), their differences into P, then S(T_i) = 4 pi sum_b kappa_abs P_b(T_i)
// per species by one warp each from the row in shared memory. The star's spectrum (the
// first block, so that its serial chain runs beside the rows) and the opacities need
// nothing of the rows: with launches of their own, as the guides below, the tables of 2
// species x 100 bins took 122 us, in two launches 83.
constexpr int kRowThreads = 128;

__global__ void __launch_bounds__(kRowThreads) k_table_rows(TableBuild tb) {
  __shared__ double edge[kMaxBins + 1];
  __shared__ double P[kMaxBins];
  const int B = tb.B, i = (int)blockIdx.x - 1;
  if (i < 0) {
    star_spectrum(tb, edge);
    return;
  }
  if (i >= tb.n_T) {
    const int b = (i - tb.n_T) * kRowThreads + threadIdx.x;
    if (b < B) opacities(tb, b);
    return;
  }
  const double T = table_T(i, tb.n_T, tb.t_min, tb.t_max);
  const double a = T > 0.0 ? kH / (kK * T) : 0.0, pref = T > 0.0 ? planck_factor(T) : 0.0;
  if (threadIdx.x == 0) tb.Tgrid[i] = T;
  for (int b = threadIdx.x; b <= B; b += kRowThreads)
    edge[b] = T > 0.0 ? planck_edge(a * tb.nu[b]) : 0.0;
  __syncthreads();
  for (int b = threadIdx.x; b < B; b += kRowThreads) {
    const double v =
        T > 0.0 ? pref * planck_between(a * tb.nu[b], edge[b], a * tb.nu[b + 1], edge[b + 1])
                : 0.0;
    P[b] = v;
    tb.P[(size_t)i * B + b] = v;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  for (int s = threadIdx.x >> 5; s < tb.S; s += kRowThreads / 32) {
    const double* ka = tb.kabs + (size_t)s * B;
    double acc = 0.0;
    for (int b = lane; b < B; b += 32) acc += ka[b] * P[b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    acc *= 4.0 * kPi;
    if (lane == 0) {
      tb.S64[(size_t)s * tb.n_T + i] = acc;
      tb.S32[(size_t)s * tb.n_T + i] = (float)acc;
    }
  }
}

// One warp per (species, interval): the normalised cumulative of
// kappa_abs(b) [P_b(T_{i+1}) - P_b(T_i)] over the bins, and the row's search guide: the
// first bin whose cumulative value exceeds k/B, k = 0 .. B-1 (at most the last bin) --
// a starting point only, the draws finish by scanning. A thread per row walking its
// bins serially, with rows B doubles apart, took 88 + 45 us for 2 species x 100 bins;
// the warp reads them coalesced and takes 21 us (the guides u_k beside them).
constexpr int kCdfWarps = 4;

__device__ __forceinline__ void u_guide(const TableBuild& tb, int idx);

__global__ void __launch_bounds__(32 * kCdfWarps) k_difference_cdfs(TableBuild tb, int n_cdf) {
  __shared__ float rows[kCdfWarps][kMaxBins];
  if ((int)blockIdx.x >= n_cdf) {
    u_guide(tb, ((int)blockIdx.x - n_cdf) * 32 * kCdfWarps + threadIdx.x);
    return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int idx = blockIdx.x * kCdfWarps + warp, nI = tb.n_T - 1, B = tb.B;
  if (idx >= tb.S * nI) return;
  const int s = idx / nI, i = idx % nI;
  const double* ka = tb.kabs + (size_t)s * B;
  const double* P0 = tb.P + (size_t)i * B;
  const double* P1 = P0 + B;
  float* out = tb.dcdf + (size_t)idx * B;
  float* row = rows[warp];
  cumulative_warp(
      B, [&](int b) { return fmax(ka[b] * (P1[b] - P0[b]), 0.0); },
      [&](int b, float c) {
        row[b] = c;
        out[b] = c;
      });
  __syncwarp();
  unsigned short* gd = tb.cdf_guide + (size_t)idx * B;
  for (int k = lane; k < B; k += 32) {
    const float thr = (float)k / (float)B;
    int lo = 0, hi = B - 1;  // the first bin above thr, or the last
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (row[mid] > thr) hi = mid; else lo = mid + 1;
    }
    gd[k] = (unsigned short)lo;
  }
}

// Per species: for u_k = exp(ln S(T_1) + k (ln S(T_last) - ln S(T_1)) / (n_T - 1)),
// the largest interval i <= n_T - 2 with S(T_i) <= u_k. One thread per (s, k).
__device__ __forceinline__ void u_guide(const TableBuild& tb, int idx) {
  if (idx >= tb.S * tb.n_T) return;
  int s = idx / tb.n_T, k = idx % tb.n_T;
  const double* S = tb.S64 + (size_t)s * tb.n_T;
  int nI = tb.n_T - 1;
  double l0 = log(S[1]), l1 = log(S[nI]);
  double u = exp(l0 + (l1 - l0) * (double)k / (double)nI);
  int lo = 0, hi = nI;  // S[lo] <= u < S[hi] (clamped at the last interval)
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (S[mid] <= u) lo = mid; else hi = mid;
  }
  tb.u_guide[idx] = lo;
}

// 1/x to 4e-15 from its FP32 value: a reciprocal there and one Newton step (the FP64 division
// is some ten operations of a pipe that does two a clock). For x well inside FP32's range.
__device__ __forceinline__ double reciprocal(float x32, double x) {
  const double r = (double)__frcp_rn(x32);
  return fma(r, fma(-x, r, 1.0), r);
}

// a < b for doubles that are not negative: their bits as integers (a compare is an FP64
// operation too)
__device__ __forceinline__ bool below(double a, double b) {
  return __double_as_longlong(a) < __double_as_longlong(b);
}

// S at temperature T by linear interpolation in T between table rows (the same
// piecewise-linear model the transport samples from), a thread per species and cell.
// A binary search of FP64 rows, then an FP64 division: 3.2e7 entries 1.46 ms, now 0.65; FP64
// operations, some twelve an entry, still bound it.
__global__ void k_frozen_u(DevGrid g, DevTables t, const float* T_frozen, float* u_frozen,
                           float t_min, float t_max) {
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c >= g.n_leaves) return;
  const int s = blockIdx.y;
  const long long idx = s * g.n_leaves + c;
  const float T32 = fmaxf(T_frozen[idx], t_min);
  const double T = (double)T32;
  const double* Tg = t.Tgrid;
  const double* S = t.S64 + (size_t)s * g.n_T;
  const int n_T = g.n_T;
  double u;
  if (!below(T, Tg[n_T - 1])) {
    u = S[n_T - 1];
  } else {
    // Tg[lo] <= T < Tg[lo + 1]: the rows from the second on are evenly spaced in ln T, so
    // start there and finish by scanning
    const float l1 = __logf(t_min), step = (__logf(t_max) - l1) / (float)(n_T - 2);
    const float k = (__logf(T32) - l1) / step + 1.0f;
    int lo = (int)fminf(fmaxf(k, 0.0f), (float)(n_T - 2));
    while (lo > 0 && below(T, Tg[lo])) --lo;
    while (lo + 2 < n_T && !below(T, Tg[lo + 1])) ++lo;
    const double dT = Tg[lo + 1] - Tg[lo];
    double w = T - Tg[lo];
    if ((float)dT > 1e-30f && (float)dT < 1e30f) {
      w *= reciprocal((float)dT, dT);  // to 4e-15; w makes up a few per cent of u at most
    } else {
      w /= dT;
    }
    u = S[lo] + w * (S[lo + 1] - S[lo]);
  }
  u_frozen[idx] = (float)u;
}

// T from n eps = M S(T): the FP64 S table's interval (guide + scan), then power-law
// (log-log) interpolation between rows; linear from T = 0 in the first interval.
//
// FP64 operations bound it (two a clock per SM): four divisions an entry before. u needs
// FP64 against the rows (they differ by a few per cent, T by less than one), but the place
// within an interval does not: differences in FP64, their quotients (of numbers well above
// rounding) in FP32, as the new T is T_i plus at most a per cent of it. Against 80 bits: 2.6e-8 RMS, 6.1e-8 at most (the
// rounding of the FP32 result; with divisions 6.4e-8 and 2.4e-7, from the quotient of
// neighbouring T in FP32).
__device__ __forceinline__ float cell_temperature(const DevTables& t, int n_T, int s, double n,
                                                  float rho_d0, int lev, unsigned& clamped) {
  if (!(n > 0.0) || !(rho_d0 > 0.0f)) return 0.0f;
  const double rho = (double)rho_d0, k = t.eps_over_V[lev] * t.d0;
  double u;
  if (rho_d0 > 1e-30f && rho_d0 < 1e30f) {
    u = n * k * reciprocal(rho_d0, rho);
  } else {
    u = n * k / rho;
  }
  const double* S = t.S64 + (size_t)s * n_T;
  const double* Tg = t.Tgrid;
  const int nI = n_T - 1;
  if (!below(u, S[nI])) {
    ++clamped;
    return (float)Tg[nI];
  }
  // interval i with S[i] <= u < S[i+1]: start from the guide of ln S (the re-emission
  // draws use the same one), finish by scanning
  const float kf = (__logf(fmaxf((float)u, 1e-30f)) - t.u_ln0[s]) * t.u_inv[s];
  int i = t.u_guide[s * n_T + (int)fminf(fmaxf(kf, 0.0f), (float)nI)];
  double Si = S[i], Sn = S[i + 1];
  while (i > 0 && below(u, Si)) {
    Sn = Si;
    Si = S[--i];
  }
  while (i + 1 < nI && !below(u, Sn)) {
    Si = Sn;
    Sn = S[++i + 1];
  }
  const double T0 = Tg[i], T1 = Tg[i + 1];
  if (i == 0 || !(Si > 0.0)) return (float)(T1 * u / Sn);
  // power law between the rows: ln(T/T_i) = ln(u/S_i) ln(T_i+1/T_i) / ln(S_i+1/S_i)
  float x = (float)(u - Si), xs = (float)(Sn - Si);
  const float S32 = (float)Si;
  if (S32 > 1e-28f && S32 < 1e30f) {
    x /= S32;
    xs /= S32;
  } else {
    x = (float)((u - Si) / Si);
    xs = (float)((Sn - Si) / Si);
  }
  const float y = log1pf(x) / log1pf(xs) * log1pf((float)(T1 - T0) / (float)T0);
  return (float)fma(T0, (double)expm1f(y), T0);
}

// Temperatures of one cell. A thread takes all its species (from s0 on in steps of s_step):
// their densities (and path-length tallies) lie side by side, a thread per species and cell
// read them in as many passes. With the arithmetic above: 8.0e6 cells of four species 0.60 ->
// 0.31 ms, 2.4e6 of two 0.20 -> 0.11.
template <int kS>
__device__ __forceinline__ void cell_temperatures(const DevGrid& g, const DevTables& t,
                                                  const unsigned long long* count, float* T_out,
                                                  const float* pathabs, long long c,
                                                  unsigned& clamped, int s0 = 0, int s_step = 1) {
  const int S = kS > 0 ? kS : g.S;
  const int lev = g.level[c];
  // absorbed energy in units of eps: the count, or the path-length tally
  const auto absorbed = [&](int s) {
    return pathabs ? (double)pathabs[tally_place(c) * tally_row(S) + s] : (double)count[s * g.n_leaves + c];
  };
  if constexpr (kS > 0) {
    double n[kS];
    float rho[kS];
#pragma unroll
    for (int s = 0; s < kS; ++s) {
      n[s] = absorbed(s);
      rho[s] = g.rho[c * kS + s];
    }
#pragma unroll
    for (int s = 0; s < kS; ++s)
      T_out[s * g.n_leaves + c] = cell_temperature(t, g.n_T, s, n[s], rho[s], lev, clamped);
  } else {
    for (int s = s0; s < S; s += s_step)
      T_out[s * g.n_leaves + c] =
          cell_temperature(t, g.n_T, s, absorbed(s), g.rho[c * S + s], lev, clamped);
  }
}

__device__ __forceinline__ void add_clamped(unsigned clamped, unsigned long long* counters) {
  clamped = __reduce_add_sync(0xffffffffu, clamped);
  if ((threadIdx.x & 31) == 0 && clamped)
    atomicAdd(&counters[kCClamped], (unsigned long long)clamped);
}

template <int kS>
__global__ void __launch_bounds__(256) k_temperatures(DevGrid g, DevTables t,
                                                      const unsigned long long* count,
                                                      float* T_out, unsigned long long* counters,
                                                      const float* pathabs) {
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  unsigned clamped = 0;
  if (c < g.n_leaves)
    cell_temperatures<kS>(g, t, count, T_out, pathabs, c, clamped, blockIdx.y, gridDim.y);
  add_clamped(clamped, counters);
}

// ---------------------------------------------------------------- batches
// All models of a batch in one launch: blockIdx.x the model, gridDim.y blocks share its
// cells. With four memsets and a temperature kernel per model, one after another, a pass
// over 24 models took 5.79 ms, with these two launches 5.50.
__device__ __forceinline__ const ModelDesc& stage_model(const ModelDesc* models) {
  __shared__ ModelDesc md;
  const int* src = reinterpret_cast<const int*>(&models[blockIdx.x]);
  for (int i = threadIdx.x; i < (int)(sizeof(ModelDesc) / sizeof(int)); i += blockDim.x)
    reinterpret_cast<int*>(&md)[i] = src[i];
  __syncthreads();
  return md;
}

template <int kS>
__global__ void __launch_bounds__(256) k_batch_temperatures(const ModelDesc* models) {
  const ModelDesc& md = stage_model(models);
  unsigned clamped = 0;
  for (long long c = blockIdx.y * 256ll + threadIdx.x; c < md.g.n_leaves; c += 256ll * gridDim.y)
    cell_temperatures<kS>(md.g, md.t, md.r.count, md.T_out, nullptr, c, clamped);
  add_clamped(clamped, md.r.counters);
}

// Counts, spectra, counters and status to zero.
__global__ void __launch_bounds__(256) k_batch_reset(const ModelDesc* models) {
  const ModelDesc& md = stage_model(models);
  const long long first = blockIdx.y * 256ll + threadIdx.x, stride = 256ll * gridDim.y;
  const long long n = md.g.S * md.g.n_leaves, n_sed = 2ll * md.g.n_dir * md.g.B;
  ulonglong2* pairs = reinterpret_cast<ulonglong2*>(md.r.count);
  for (long long i = first; i < n / 2; i += stride) pairs[i] = make_ulonglong2(0ull, 0ull);
  if (first == 0 && (n & 1)) md.r.count[n - 1] = 0ull;
  for (long long i = first; i < n_sed; i += stride) md.r.sed[i] = 0ull;
  if (first < kNumCounters) md.r.counters[first] = 0ull;
  if (first == 0) *md.r.status = 0u;
}

// Path-length tallies, species within a cell adjacent, to one array per species: a block of
// rows is a 64 x 64 transposition (tally_place), done in tiles of 32 x 32 through shared memory
// so that reads and writes are whole sectors, kV species at a time. 8.0e6 cells, us, a cell per
// thread and in tiles: one species 33 and 12, two 60 and 25, four 119 and 42 (51 with kV = 4).
constexpr int kTile = 32, kTileRows = 8;
constexpr int kTilesAcross = (1 << kTallyBits) / kTile;

template <int kV>
__global__ void __launch_bounds__(kTile * kTileRows) k_tally_out(const float* pathabs,
                                                                 long long N, int S, float* out) {
  struct alignas(4 * kV) Vec {
    float v[kV];
  };
  __shared__ float tile[kV][kTile][kTile + 1];
  const int x = threadIdx.x & (kTile - 1), y = threadIdx.x / kTile;
  const int t = blockIdx.x % (kTilesAcross * kTilesAcross);
  const long long first = (long long)(blockIdx.x / (kTilesAcross * kTilesAcross)) * kTallyBlock;
  const int a0 = t % kTilesAcross * kTile, b0 = t / kTilesAcross * kTile;
  const int row = tally_row(S);  // a multiple of kV
  for (int s0 = 0; s0 < S; s0 += kV) {
#pragma unroll
    for (int i = y; i < kTile; i += kTileRows) {  // place first + (b0 + i) 64 + a0 + x
      const Vec r = *reinterpret_cast<const Vec*>(
          pathabs + (size_t)(first + ((b0 + i) << kTallyBits) + a0 + x) * row + s0);
#pragma unroll
      for (int v = 0; v < kV; ++v) tile[v][i][x] = r.v[v];
    }
    __syncthreads();
#pragma unroll
    for (int i = y; i < kTile; i += kTileRows) {
      const long long leaf = first + ((a0 + i) << kTallyBits) + b0 + x;
#pragma unroll
      for (int v = 0; v < kV; ++v)
        if (leaf < N && s0 + v < S) out[(size_t)(s0 + v) * N + leaf] = tile[v][x][i];
    }
    __syncthreads();
  }
}

inline unsigned nblk(long long n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

cudaError_t launch_build_tables(const TableBuild& tb, cudaStream_t s) {
  k_table_rows<<<1 + (unsigned)tb.n_T + nblk(tb.B, kRowThreads), kRowThreads, 0, s>>>(tb);
  // the guides' blocks after those of the rows
  const unsigned n_cdf = nblk((long long)tb.S * (tb.n_T - 1), kCdfWarps);
  k_difference_cdfs<<<n_cdf + nblk((long long)tb.S * tb.n_T, 32 * kCdfWarps), 32 * kCdfWarps, 0,
                      s>>>(tb, (int)n_cdf);
  return cudaGetLastError();
}

cudaError_t launch_frozen_u(const DevGrid& g, const DevTables& t, const float* T_frozen,
                            float* u_frozen, float t_min, float t_max, cudaStream_t s) {
  const dim3 grid(nblk(g.n_leaves, 256), (unsigned)g.S);
  k_frozen_u<<<grid, 256, 0, s>>>(g, t, T_frozen, u_frozen, t_min, t_max);
  return cudaGetLastError();
}

cudaError_t launch_tally_out(const DevGrid& g, const float* pathabs, float* out,
                             cudaStream_t s) {
  const long long blocks = (g.n_leaves + kTallyBlock - 1) / kTallyBlock;
  const auto kernel = g.S == 1 ? k_tally_out<1> : k_tally_out<2>;
  kernel<<<(unsigned)(blocks * kTilesAcross * kTilesAcross), kTile * kTileRows, 0, s>>>(
      pathabs, g.n_leaves, g.S, out);
  return cudaGetLastError();
}

cudaError_t launch_temperatures(const DevGrid& g, const DevTables& t,
                                const unsigned long long* count, float* T_out,
                                unsigned long long* counters, cudaStream_t s,
                                const float* pathabs) {
  // A thread per cell where a cell's species are one vector and the cells fill the chip, else a
  // thread per species and cell. Cell and species, us: two species, 512 cells 8.2 and 6.2,
  // 2.6e5 26.7 and 26.7; four, 512 cells 11.4 and 6.2, 2.6e5 31.2 and 30.0, 8.8e5 78 and 84;
  // eight (no vector), 512 cells 18.5 and 6.2, 8.8e5 109 and 108.
  const bool cells = (g.S == 2 || g.S == 4) && g.n_leaves > 1 << 18;
  const auto kernel = !cells ? k_temperatures<0> : (g.S == 2 ? k_temperatures<2>
                                                             : k_temperatures<4>);
  kernel<<<dim3(nblk(g.n_leaves, 256), cells ? 1 : (unsigned)g.S), 256, 0, s>>>(
      g, t, count, T_out, counters, pathabs);
  return cudaGetLastError();
}

static dim3 batch_grid(int n_models, long long max_cells) {
  const long long blocks = (max_cells + 255) / 256;
  return dim3((unsigned)n_models, (unsigned)(blocks < 1024 ? blocks : 1024));
}

cudaError_t launch_batch_temperatures(const ModelDesc* models, int n_models, long long max_cells,
                                      int s_fixed, cudaStream_t s) {
  const auto kernel = s_fixed == 2 ? k_batch_temperatures<2>
                                   : (s_fixed == 4 ? k_batch_temperatures<4>
                                                   : k_batch_temperatures<0>);
  kernel<<<batch_grid(n_models, max_cells), 256, 0, s>>>(models);
  return cudaGetLastError();
}

cudaError_t launch_batch_reset(const ModelDesc* models, int n_models, long long max_cells,
                               cudaStream_t s) {
  k_batch_reset<<<batch_grid(n_models, max_cells), 256, 0, s>>>(models);
  return cudaGetLastError();
}

}  // namespace rt
