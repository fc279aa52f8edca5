// rt_pah.cu -- transiently heated PAH molecules on the device: FP64 level tables,
// template re-emission spectra, and the exact steady-state emission per cell.
//
// Thermal-discrete steady state (Guhathakurta & Draine 1989): internal-energy
// levels E_f = f dE, f = 0 .. M-1; absorbing a photon of energy e moves a molecule
// from E_i up to E_i + e, split between the two levels around it so the energy is
// kept (uniform levels: e/dE = q + w gives levels i+q and i+q+1 with weights 1-w and
// w); cooling is continuous at L(E) = 4 pi sum_b sigma_b P_b(T(E)), a step to the
// level below at rate C_f = L_f / dE. The upward probability flux across each level
// boundary equals C_f P_f, so the populations follow level by level. The molecule
// then emits sum_f P_f 4 pi sigma_b P_b(T_f) in bin b.

#include "rt_internal.h"
#include "rt_planck.cuh"

#include <math.h>

namespace rt {
namespace {

using namespace planck;

constexpr double kHh = 6.62607015e-27;

// The level emission table: levels in pairs, [pair][bin][2], bins padded to whole groups of
// four -- a bin's values at two levels are one operand of a packed FP32 multiply-add.
__host__ __device__ constexpr int pad4(int b) { return (b + 3) & ~3; }
__host__ __device__ constexpr size_t level_at(int f, int b, int B) {
  return ((size_t)(f >> 1) * pad4(B) + b) * 2 + (f & 1);
}

__device__ double heat_content(double T, const PahSpec& sp) {
  if (!(T > 0.0)) return 0.0;
  double e = 0.0;
  for (int i = 0; i < sp.n_groups; ++i) {
    double x = sp.theta[i] / T;
    if (x < 700.0) e += sp.n_modes[i] * kK * sp.theta[i] / expm1(x);
  }
  return e;
}

__device__ double temperature_of(double E, const PahSpec& sp) {
  if (!(E > 0.0)) return 0.0;
  double lo = 1e-3, hi = 10.0;
  while (heat_content(hi, sp) < E && hi < 1e9) hi *= 2.0;
  for (int it = 0; it < 200; ++it) {
    double mid = sqrt(lo * hi);
    if (heat_content(mid, sp) < E) lo = mid; else hi = mid;
    if (hi / lo - 1.0 < 1e-14) break;
  }
  return sqrt(lo * hi);
}

// The temperature at heat content E: an FP32 bisection (cheap here: FP64 runs at 1/64 of
// the FP32 rate) gives a start good to about 1e-6, from which Newton's method in FP64
// converges to the last bits in two steps; where it does not (a start out of the FP32
// range), the FP64 bisection. One thread; the bisection alone takes 50 FP64 evaluations.
__device__ double level_temperature(double E, const PahSpec& sp) {
  if (!(E > 0.0)) return 0.0;
  // FP32: heat contents relative to E, ln T in [ln 1e-3, ln 1e9]
  float w[kMaxModeGroups], th[kMaxModeGroups];
#pragma unroll
  for (int i = 0; i < kMaxModeGroups; ++i) {
    w[i] = i < sp.n_groups ? (float)(sp.n_modes[i] * kK * sp.theta[i] / E) : 0.0f;
    th[i] = i < sp.n_groups ? (float)sp.theta[i] : 1.0f;
  }
  float lo = -6.9077554f, hi = 20.723266f;
  for (int it = 0; it < 25; ++it) {
    const float mid = 0.5f * (lo + hi), rT = expf(-mid);
    float e = 0.0f;
#pragma unroll
    for (int i = 0; i < kMaxModeGroups; ++i) e += w[i] / expm1f(fminf(th[i] * rT, 80.0f));
    if (e < 1.0f) lo = mid; else hi = mid;
  }
  double T = exp(0.5 * ((double)lo + (double)hi));
  for (int it = 0; it < 6; ++it) {
    double e = 0.0, de = 0.0;  // heat content and T times its derivative
    for (int i = 0; i < sp.n_groups; ++i) {
      const double x = sp.theta[i] / T;
      if (x < 700.0) {
        const double m = 1.0 / expm1(x), u = sp.n_modes[i] * kK * sp.theta[i] * m;
        e += u;
        de += u * x * (1.0 + m);
      }
    }
    const double step = (E - e) / de;
    if (!(fabs(step) < 0.1)) break;
    T += T * step;
    if (fabs(step) < 1e-9) return T;  // the next step would be below 1e-16
  }
  return temperature_of(E, sp);
}

// one thread per (PAH, level): temperature of the level
__global__ void k_pah_temps(PahBuild pb) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= pb.n_pah * pb.M) return;
  const int p = idx / pb.M, f = idx % pb.M;
  pb.T[idx] = level_temperature(f * pb.dE[p], pb.spec[p]);
}

// one warp per (PAH, level): cooling rate (FP64) and emission spectrum per bin (stored
// FP32). A thread per level doing its bins one after another, the temperature by FP64
// bisection, took 20 ms for 2 x 400 levels and 200 bins; this takes 0.05 ms.
__global__ void k_pah_levels(PahBuild pb) {
  const int idx = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (idx >= pb.n_pah * pb.M) return;
  const int p = idx / pb.M, f = idx % pb.M;
  const double* sig = pb.sigma + (size_t)p * pb.B;
  float* s = pb.s + p * level_at(pad4(pb.M), 0, pb.B);
  if (lane < pad4(pb.B) - pb.B) s[level_at(f, pb.B + lane, pb.B)] = 0.0f;
  if (f == pb.M - 1)  // zero levels up to whole groups of four
    for (int z = pb.M; z < pad4(pb.M); ++z)
      for (int b = lane; b < pad4(pb.B); b += 32) s[level_at(z, b, pb.B)] = 0.0f;
  double L = 0.0;
  planck::planck_bins_warp(pb.nu, pb.B, pb.T[idx], [&](int b, double v) {
    v *= 4.0 * kPi * sig[b];
    s[level_at(f, b, pb.B)] = (float)v;
    L += v;
  });
  for (int o = 16; o > 0; o >>= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
  if (lane == 0) pb.L[idx] = L;
}

// coarse photon energies e_k = h sqrt(nu_lo nu_hi) over each coarse bin's range,
// and their split q_k + w_k = e_k / dE for every PAH
__global__ void k_pah_coarse(PahBuild pb) {
  int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= pb.n_pah * pb.K) return;
  int p = idx / pb.K, k = idx % pb.K;
  int b0 = (k * pb.B + pb.K - 1) / pb.K;          // first fine bin with floor(b K/B) == k
  int b1 = ((k + 1) * pb.B + pb.K - 1) / pb.K - 1;  // last one
  double e = kHh * sqrt(pb.nu[b0] * pb.nu[b1 + 1]);
  if (p == 0) pb.e_k[k] = e;
  double x = e / pb.dE[p];
  double q = floor(x);
  pb.q_k[idx] = (int)q;
  pb.w_k[idx] = x - q;
}

// For the per-cell solution: FP32 copies of c_f = L_f / dE, w_k and e_k, and for each
// distance d the number of coarse bins whose photons span fewer than d levels (q_k < d; the
// q_k rise with k)
__global__ void k_pah_f32(PahBuild pb) {
  int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx < pb.n_pah * pb.M) {
    const float c = (float)(pb.L[idx] / pb.dE[idx / pb.M]);
    pb.c_f[idx] = c > 0.0f ? c : 0.0f;
  }
  if (idx < pb.n_pah * pb.K) pb.w_f[idx] = (float)pb.w_k[idx];
  if (idx < pb.K) pb.e_f[idx] = (float)pb.e_k[idx];
  if (idx < pb.n_pah * (pb.M + 1)) {
    const int p = idx / (pb.M + 1), d = idx % (pb.M + 1);
    int k = 0;
    while (k < pb.K && pb.q_k[p * pb.K + k] < d) ++k;
    pb.first_k[idx] = (unsigned char)k;
  }
}

// Level populations of PAH p for absorption rates R[k] (smem, per molecule per
// second), one warp; P and D are this warp's shared-memory arrays of M doubles.
// Returns the emitted power sum_f P_f L_f of the normalised populations in P.
__device__ double solve_levels(const PahTables& t, int p, const double* R, double* P,
                               double* D) {
  const int lane = threadIdx.x & 31;
  const int M = t.M, K = t.K;
  const double dE = t.dE[p];
  const int* q = t.q_k + p * K;
  const double* w = t.w_k + p * K;
  const double* L = t.L + (size_t)p * M;
  for (int i = lane; i < M; i += 32) {
    D[i] = 0.0;
    P[i] = 0.0;
  }
  __syncwarp();
  double up = 0.0;
  // scatter level i's absorptions into D; returns this lane's upward rate
  auto scatter = [&](int i, double Pi) {
    double u = 0.0;
    for (int k = lane; k < K; k += 32) {
      double r = R[k];
      if (!(r > 0.0)) continue;
      int f = i + q[k];
      double wk = w[k];
      if (f >= M - 1) {
        f = M - 1;
        wk = 0.0;
      }
      if (f > i) {
        atomicAdd(&D[f], Pi * r * (1.0 - wk));
        u += r * (1.0 - wk);
      }
      if (wk > 0.0 && f + 1 < M) {
        atomicAdd(&D[f + 1], Pi * r * wk);
        u += r * wk;
      }
    }
    return u;
  };
  double P0 = 1.0;
  if (lane == 0) P[0] = P0;
  up = scatter(0, P0);
  for (int o = 16; o > 0; o >>= 1) up += __shfl_xor_sync(0xffffffffu, up, o);
  double F = P0 * up;
  for (int f = 1; f < M; ++f) {
    __syncwarp();
    double C = L[f] / dE;
    double Pf = C > 0.0 ? F / C : 0.0;
    if (lane == 0) P[f] = Pf;
    double u = scatter(f, Pf);
    for (int o = 16; o > 0; o >>= 1) u += __shfl_xor_sync(0xffffffffu, u, o);
    __syncwarp();
    F = fmax(F - D[f] + Pf * u, 0.0);
    if (Pf > 1e250) {  // keep the numbers finite
      __syncwarp();
      for (int i = lane; i < M; i += 32) {
        P[i] *= 1e-250;
        D[i] *= 1e-250;
      }
      F *= 1e-250;
    }
  }
  __syncwarp();
  double tot = 0.0, em = 0.0;
  for (int i = lane; i < M; i += 32) tot += P[i];
  for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
  __syncwarp();
  for (int i = lane; i < M; i += 32) {
    P[i] /= tot;
    em += P[i] * L[i];
  }
  for (int o = 16; o > 0; o >>= 1) em += __shfl_xor_sync(0xffffffffu, em, o);
  __syncwarp();
  return em;
}

// Template re-emission spectra: one warp per PAH, heated by the source's blackbody
// at bolometric flux pb.f_ref inside the frequency grid.
__global__ void k_pah_template(PahTables t, PahBuild pb) {
  extern __shared__ double sm[];
  const int p = blockIdx.x;
  const int lane = threadIdx.x;
  double* R = sm;            // [K]
  double* P = R + t.K;       // [M]
  double* D = P + t.M;       // [M]
  const double* sig = pb.sigma + (size_t)p * pb.B;
  // stellar flux per fine bin, summed into coarse photon rates
  double tot = 0.0;
  for (int b = lane; b < pb.B; b += 32) tot += planck_bin(pb.nu[b], pb.nu[b + 1], pb.T_star);
  for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
  for (int k = lane; k < t.K; k += 32) R[k] = 0.0;
  __syncwarp();
  for (int b = lane; b < pb.B; b += 32) {
    double fb = pb.f_ref * planck_bin(pb.nu[b], pb.nu[b + 1], pb.T_star) / tot;
    int k = (int)(((long long)b * t.K) / pb.B);
    atomicAdd(&R[k], fb * sig[b] / t.e_k[k]);
  }
  __syncwarp();
  solve_levels(t, p, R, P, D);
  // J_b = sum_f P_f s_fb, then its normalised cumulative
  float* cdf = pb.template_cdf + (size_t)p * pb.B;
  double run = 0.0;
  for (int b0 = 0; b0 < pb.B; b0 += 32) {
    int b = b0 + lane;
    double j = 0.0;
    if (b < pb.B)
      for (int f = 0; f < t.M; ++f) j += P[f] * (double)t.s[p * level_at(pad4(t.M), 0, pb.B) + level_at(f, b, pb.B)];
    // inclusive scan over the 32 lanes
    double x = j;
    for (int o = 1; o < 32; o <<= 1) {
      double y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (b < pb.B) cdf[b] = (float)(run + x);  // unnormalised for now
    run += __shfl_sync(0xffffffffu, x, 31);
  }
  __syncwarp();
  for (int b = lane; b < pb.B; b += 32) cdf[b] = run > 0.0 ? (float)((double)cdf[b] / run) : 1.0f;
  __syncwarp();
  if (lane == 0) cdf[pb.B - 1] = 1.0f;
}

// The same steady state in FP32, for the per-cell solutions: a group of 8 lanes per cell (4
// cells per warp; a group without a cell solves a zero rate vector). The levels are
// uniform, so the rate from level i to the levels at or above f depends on f - i alone:
// G(d) = sum over coarse bins of the rate landing d or more levels up (an absorption split
// between i + q_k and i + q_k + 1, or cut at the top level, counts alike for every f <= M -
// 1). The upward flux across the boundary below f is then F_f = sum_{d >= 1} G(d) P_{f-d}
// -- the quantity the carried recursion forms, here as a dot product of positive terms,
// with no cancellation in FP32 (about 1e-7 relative on every level that matters) and no
// scatter. P_f = F_f / C_f.
//
// A triangular Toeplitz solve, done in blocks of 8 levels. What a block below gives to a
// block's 8 fluxes is a small convolution: 64 products from its 8 populations and 15 rates.
// The 8 lanes share the distances between the blocks, n each (n odd, so that their reads of
// the populations fall on different banks): a lane's rates are the same for every block and
// stay in registers, and a pair of blocks costs two 16-byte shared-memory reads. A
// transposing butterfly leaves lane i with flux i, and 8 short steps (divide, broadcast,
// multiply-add) solve the block itself.
//
// One level at a time (a dot product over 4 lanes, two 4-byte reads a product, two
// shuffles, a division and a barrier per level) 5.0e4 cells, two PAHs and 200 bins took
// 3.9 ms with their emission, now 1.23 ms, about half of it here. What bounds it now is
// latency: 16 warps an SM, 44 % of the issue slots used.
//
// The populations of a cell are split into the lower and upper halves of the 8-blocks
// (element f at half (f >> 2) & 1, place 4 (f >> 3) + (f & 3)), so that 16-byte reads of
// consecutive blocks fall on consecutive addresses; the rates use the same memory before
// the populations do. Populations are kept below 1e20 by rescaling (the normalised result
// is unchanged). Leaves the unnormalised populations in P and returns this lane's part of
// their sum.
struct Halves {
  float* lo;
  float* hi;
  __device__ __forceinline__ Halves(float* base, int nb) : lo(base), hi(base + 4 * nb) {}
  __device__ __forceinline__ float& at(int f) const {
    return ((f & 4) ? hi : lo)[4 * (f >> 3) + (f & 3)];
  }
  __device__ __forceinline__ void read(int blk, float* v) const {
    const float4 a = reinterpret_cast<const float4*>(lo)[blk];
    const float4 b = reinterpret_cast<const float4*>(hi)[blk];
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  }
  __device__ __forceinline__ void write(int blk, const float* v) const {
    reinterpret_cast<float4*>(lo)[blk] = make_float4(v[0], v[1], v[2], v[3]);
    reinterpret_cast<float4*>(hi)[blk] = make_float4(v[4], v[5], v[6], v[7]);
  }
};

constexpr float kTopPopulation = 1e20f;

// two FP32 multiply-adds in one instruction, and the sum of a pair
__device__ __forceinline__ void fma2(unsigned long long& acc, unsigned long long a,
                                     unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ float sum2(unsigned long long a) {
  return __uint_as_float((unsigned)a) + __uint_as_float((unsigned)(a >> 32));
}

// G of a cell from its absorbed counts. All coarse bins whose photons span d levels or more
// land d or more levels up whole, those that span between d - 1 and d with the part w of
// their split: G(d) = sum_{k >= first(d)} R_k + sum_{q_k = d - 1} w_k R_k, a suffix sum over
// the bins and a short sum (no scatter into G and no atomics). tmp: 2 x 72 floats of the
// cell. Returns the largest d with a rate; *any whether anything was absorbed. All lanes of
// the warp; cnt null for a group without a cell.
__device__ __forceinline__ int cell_rates(const PahTables& t, int p, const unsigned* cnt,
                                          float scale, const Halves& G, int nb, float* tmp,
                                          bool* any) {
  const int l = threadIdx.x & 7, K = t.K;
  float* suffix = tmp;       // [K + 1]
  float* split = tmp + 72;   // [K] w_k R_k
  const float* wf = t.w_f + p * K;
  float r[8];  // bins 8 l ..
  unsigned seen = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int k = 8 * l + i;
    const unsigned v = cnt && k < K ? __ldg(&cnt[k]) : 0u;
    seen |= v;
    r[i] = v ? (float)v * scale / __ldg(&t.e_f[k]) : 0.0f;
  }
  int top = -1;  // highest bin with a rate
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    if (r[i] > 0.0f) top = 8 * l + i;
    split[8 * l + i] = r[i] > 0.0f ? r[i] * __ldg(&wf[8 * l + i]) : 0.0f;
  }
#pragma unroll
  for (int i = 6; i >= 0; --i) r[i] += r[i + 1];
  float above = r[0];  // inclusive sum over this and the higher lanes
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    const float u = __shfl_down_sync(0xffffffffu, above, o, 8);
    if (l + o < 8) above += u;
  }
  above = __shfl_down_sync(0xffffffffu, above, 1, 8);
  if (l == 7) above = 0.0f;
#pragma unroll
  for (int i = 0; i < 8; ++i) suffix[8 * l + i] = r[i] + above;
  if (l == 7) suffix[64] = 0.0f;
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
    seen |= __shfl_xor_sync(0xffffffffu, seen, o);
    top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
  }
  *any = seen != 0;
  const int dmax = top >= 0 ? min(__ldg(&t.q_k[p * K + top]) + 1, t.M - 1) : 0;
  const float zero[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
  for (int b = l; b < nb; b += 8) G.write(b, zero);
  __syncwarp();
  const unsigned char* first = t.first_k + p * (t.M + 1);
  for (int d = 1 + l; d <= dmax; d += 8) {
    const int k1 = __ldg(&first[d]);
    float v = suffix[k1];
    for (int k = __ldg(&first[d - 1]); k < k1; ++k) v += split[k];
    G.at(d) = v;
  }
  __syncwarp();
  return dmax;
}

// P may be the memory of G. kNear: the lane's rates in registers, blocks 8 kNear apart at
// most; 0: any distance, the rates read from G, which then is memory of its own.
template <int kNear>
__device__ float solve_levels_f32(const float* cf, int M, const Halves& P, const Halves& G,
                                  int dmax) {
  const int l = threadIdx.x & 7;
  const unsigned group = 0xffu << (threadIdx.x & 24);
  const int nb = (M + 7) >> 3, reach = (dmax + 7) >> 3;
  float near[7];  // G(l - i): what level i of a block gives to this lane's
#pragma unroll
  for (int i = 0; i < 7; ++i) near[i] = l > i ? G.at(l - i) : 0.0f;
  float g[kNear > 0 ? 8 * (kNear + 1) : 16];
  if constexpr (kNear > 0) {
#pragma unroll
    for (int b = 0; b <= kNear; ++b) {
      if (l * kNear + b < nb) {
        G.read(l * kNear + b, g + 8 * b);
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) g[8 * b + i] = 0.0f;
      }
    }
    __syncwarp();
  }
  float tot = 0.0f;
  for (int fb = 0; fb < nb; ++fb) {
    const int f = 8 * fb + l;
    const float C = f < M ? __ldg(&cf[f]) : 0.0f;
    float F[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) F[i] = 0.0f;
    auto add = [&](int jb, const float* w) {  // w: rates at 8 (fb - jb - 1) ..
      float p[8];
      P.read(jb, p);
#pragma unroll
      for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int i = 0; i < 8; ++i) F[i] = fmaf(w[8 + i - j], p[j], F[i]);
    };
    if constexpr (kNear > 0) {
#pragma unroll
      for (int m = 0; m < kNear; ++m) {
        const int jb = fb - 1 - l * kNear - m;
        if (jb >= 0) add(jb, g + 8 * m);
      }
    } else {
      for (int jb = max(0, fb - reach) + l; jb < fb; jb += 8) {
        G.read(fb - jb - 1, g);
        G.read(fb - jb, g + 8);
        add(jb, g);
      }
    }
    // lane i receives flux i
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      const bool hi = (l & o) != 0;
#pragma unroll
      for (int i = 0; i < o; ++i) {
        const float send = hi ? F[i] : F[i + o], keep = hi ? F[i + o] : F[i];
        F[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    }
    // the sum within the block carries its rounding errors along (lost), or its seven
    // roundings a level would double the error of the whole solution
    float flux = F[0], lost = 0.0f, own = 0.0f;
    const float rC = C > 0.0f ? 1.0f / C : 0.0f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      // flux / C: product with the reciprocal, corrected once
      const float sum = flux + lost;
      float q = sum * rC;
      q = C > 0.0f ? fmaf(fmaf(-q, C, sum), rC, q) : 0.0f;
      if (fb == 0 && i == 0) q = 1.0f;
      float pi = __shfl_sync(0xffffffffu, q, i, 8);
      if (!(pi <= kTopPopulation)) {
        const float sc = __shfl_sync(group, (kTopPopulation * C) / sum, i, 8);
        pi = kTopPopulation;
        if (sc >= 1.0f) {  // the reciprocal of a rate below 3e-39 (the coldest levels) overflowed
          pi = kTopPopulation / sc;
        } else {  // rescale what there is so that this level is 1e20
          for (int jb = l; jb < fb; jb += 8) {
            float p[8];
            P.read(jb, p);
#pragma unroll
            for (int k = 0; k < 8; ++k) p[k] *= sc;
            P.write(jb, p);
          }
          __syncwarp(group);
          own *= sc;
          flux *= sc;
          lost *= sc;
          tot *= sc;
        }
      }
      if (l == i) own = pi;
      if (i < 7) {
        const float next = fmaf(near[i], pi, flux);
        lost += fmaf(near[i], pi, flux - next);
        flux = next;
      }
    }
    P.at(f) = own;
    tot += own;
    __syncwarp();
  }
  return tot;
}

// 1 / x to FP64 precision from the FP32 reciprocal by one Newton step (the FP64 division is
// some thirty operations at 1/64 of the FP32 rate).
__device__ __forceinline__ double reciprocal(float x) {
  if (!(x > 1e-37f && x < 1e37f)) return 1.0 / (double)x;
  const double r = (double)(1.0f / x);
  return fma(r, fma(-(double)x, r, 1.0), r);
}

// A positive FP64 factor as two FP32 parts of its mantissa and two powers of two, which
// scale an FP32 number as the FP64 product rounded to FP32 would (the factor may lie
// outside the FP32 range).
struct Scale {
  float hi, lo, s1, s2;
};

__device__ __forceinline__ Scale split_scale(double f) {
  const long long bits = __double_as_longlong(f);
  const int e = (int)((bits >> 52) & 0x7ff) - 1023, e1 = e / 2;
  const double m = __longlong_as_double((bits & 0x800fffffffffffffll) | 0x3ff0000000000000ll);
  Scale s;
  s.hi = (float)m;
  s.lo = (float)(m - (double)s.hi);
  s.s1 = __int_as_float(min(max(e1 + 127, 1), 254) << 23);
  s.s2 = __int_as_float(min(max(e - e1 + 127, 1), 254) << 23);
  return s;
}

__device__ __forceinline__ float scaled(float x, const Scale& s) {
  return fmaf(x, s.hi, x * s.lo) * s.s1 * s.s2;
}

// Per PAH and refinement level: molecules in a cell of unit stored density (density times
// base-cube edge), and eps over them.
struct CellScales {
  double molecules[kMaxPah][kMaxLevels];
  double eps_per_molecule[kMaxPah][kMaxLevels];
  double size_feature[kMaxPah];  // log10(N_C) - 2
};

// Exact emission of cells [first, first + n): a group of 8 lanes per cell solves the level
// populations (all PAH species in turn); the block's cells then form their emission
// together, J_cb = sum_f P_cf s_fb, in tiles of 8 cells x 4 bins per thread (a row of the
// level table s, read from L2, serves every cell of the block; FP32 issue bounds it).
// j_out[c][b] = sum over PAH of N_mol sum_f P_f s_fb (erg/s per bin). N_mol can exceed the
// FP32 range: its products are formed in FP64, or in FP32 parts that keep its precision.
// Shared memory of a cell (floats): its populations, apart from them its rates where the
// level grid is longer than the register form spans (8 lanes x 7 blocks), and the coarse
// bins' sums.
constexpr int kNearMost = 7;
__host__ __device__ constexpr bool rates_apart(int M) { return M > 64 * kNearMost; }
__host__ __device__ constexpr int exact_cell_floats(int M) {
  return (rates_apart(M) ? 16 : 8) * ((M + 7) / 8) + 4 + 144;
}

constexpr int kCells = 8;  // per block of two warps

template <int kMinBlocks>
__global__ void __launch_bounds__(8 * kCells, kMinBlocks)
    k_pah_exact(DevGrid g, PahTables t, const __grid_constant__ CellScales sc,
                const unsigned* pahabs, long long first, long long n, float* j_out, int pah_only, const int* list,
                const int* cell_of_row) {
  extern __shared__ __align__(16) float smf[];
  __shared__ Scale s_norm[kCells];     // N_mol / sum_f P_f, 0 without a solution
  __shared__ long long s_row[kCells];  // row of j_out
  const int slot = threadIdx.x >> 3, l = threadIdx.x & 7;
  const int nb = (t.M + 7) >> 3, CS = exact_cell_floats(t.M);
  float* own = smf + (size_t)slot * CS;
  const Halves P(own, nb), G(own + (rates_apart(t.M) ? 8 * nb : 0), nb);
  const long long i = (long long)blockIdx.x * kCells + slot;
  // row of j_out; the cell is first + row, or first + cell_of_row[row] when the
  // output rows are a compact list of cells
  const long long c = i < n ? (list ? (long long)list[i] : i) : -1;
  const long long cell = i < n ? first + (cell_of_row ? (long long)cell_of_row[c] : c) : -1;
  if (l == 0) s_row[slot] = c;
  const int lev = i < n ? g.level[cell] : 0;
  const int quads = pad4(g.B) >> 2, tiles = quads * (kCells / 8);
  for (int p = 0, done = 0; p < t.n_pah; ++p) {
    if (pah_only >= 0 && p != pah_only) continue;
    // molecules, and the absorption rate per molecule of a count of 1 erg: eps / N_mol
    const float rho = i < n ? g.rho[cell * g.S + t.species[p]] : 0.0f;
    const double n_mol = (double)rho * sc.molecules[p][lev];
    const float scale = rho > 0.0f ? (float)(sc.eps_per_molecule[p][lev] * reciprocal(rho)) : 0.0f;
    bool any;
    const int dmax = cell_rates(
        t, p, i < n ? pahabs + ((size_t)p * g.n_leaves + cell) * t.K : nullptr, scale, G, nb,
        own + CS - 144, &any);
    // every group of the warp solves (a zero rate vector where there is nothing to
    // solve), so the warp stays converged for its shuffles
    Scale norm{};
    if (__any_sync(0xffffffffu, any && n_mol > 0.0)) {
      const float* cf = t.c_f + (size_t)p * t.M;
      // the furthest block any photon reaches from (not this cell's: a cell's sums are taken
      // in the same order whatever cells share its warp)
      const int far = (min(__ldg(&t.q_k[p * t.K + t.K - 1]) + 1, t.M - 1) + 7) >> 3;
      float tot;
      if (far <= 8)
        tot = solve_levels_f32<1>(cf, t.M, P, G, dmax);
      else if (far <= 24)
        tot = solve_levels_f32<3>(cf, t.M, P, G, dmax);
      else if (far <= 8 * kNearMost)
        tot = solve_levels_f32<kNearMost>(cf, t.M, P, G, dmax);
      else
        tot = solve_levels_f32<0>(cf, t.M, P, G, dmax);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
      if (any && n_mol > 0.0) norm = split_scale(n_mol * reciprocal(tot));
    } else if (rates_apart(t.M)) {
      const float zero[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
      for (int b = l; b < nb; b += 8) P.write(b, zero);
    }
    if (l == 0) s_norm[slot] = norm;
    __syncthreads();
    for (int tile = threadIdx.x; tile < tiles; tile += 8 * kCells) {
      // bins b, b + 1 and, half the bins further, b + h, b + h + 1: 16 bytes side by side
      // between neighbouring lanes in each of the loads
      const int c0 = (tile / quads) * 8, b = (tile % quads) * 2, h = 2 * quads;
      // per cell and bin the sums over the even and the odd levels
      unsigned long long acc[8][4];
#pragma unroll
      for (int w = 0; w < 8; ++w)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[w][u] = 0ull;
      const ulonglong2* sp = reinterpret_cast<const ulonglong2*>(
          t.s + p * level_at(pad4(t.M), 0, g.B) + 2 * b);
      for (int f0 = 0; f0 < t.M; f0 += 4) {
        ulonglong2 sf[2][2];  // two pairs of levels x four bins
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          sf[u][0] = __ldg(sp + (size_t)(f0 / 2 + u) * 2 * quads);
          sf[u][1] = __ldg(sp + (size_t)(f0 / 2 + u) * 2 * quads + quads);
        }
        const float* at = smf + ((f0 & 4) ? 4 * nb : 0) + 4 * (f0 >> 3);
#pragma unroll
        for (int w = 0; w < 8; ++w) {
          const ulonglong2 pf =
              *reinterpret_cast<const ulonglong2*>(at + (size_t)(c0 + w) * CS);
          const unsigned long long pv[2] = {pf.x, pf.y};
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            fma2(acc[w][0], pv[u], sf[u][0].x);
            fma2(acc[w][1], pv[u], sf[u][0].y);
            fma2(acc[w][2], pv[u], sf[u][1].x);
            fma2(acc[w][3], pv[u], sf[u][1].y);
          }
        }
      }
#pragma unroll
      for (int w = 0; w < 8; ++w) {
        const long long row = s_row[c0 + w];
        if (row < 0) continue;
        const Scale nw = s_norm[c0 + w];
        float* j = j_out + (size_t)row * g.B;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int bu = b + (u & 1) + (u < 2 ? 0 : h);
          const float v = scaled(sum2(acc[w][u]), nw);
          if (bu < g.B) j[bu] = done ? j[bu] + v : v;
        }
      }
    }
    done = 1;
    __syncthreads();
  }
}

// Surrogate features of n_pah PAHs from `pah0` on in cells [first, first + n): the shape of
// the absorbed spectrum, x_k = ln(a_k + 1e-4)/4.6 + 1 with a_k the fraction of the absorbed
// photons in coarse bin k; the absorbed power per molecule,
// x_K = (log10(P_abs / N_mol) + 12) / 4; the size, x_K+1 = log10(N_C) - 2. Rows p n + c of X
// [n_pah n][K + 2]; p_abs[p n + c] = absorbed power of the cell's PAH (erg/s), 0 without
// absorptions; power[p n + c] (may be null) = x_K. A warp takes 32 rows: counts and features
// coalesced, a row at a time; then the FP64 logarithms of all 32 at once, a lane each (FP64
// runs at 1/64 rate: with a warp per row, one lane's logarithms, they took 0.37 ms for
// 5.5e4 rows; a thread per row, its counts uncoalesced, 0.09 ms; this 0.026).
__global__ void __launch_bounds__(64) k_pah_features(DevGrid g, PahTables t,
                                                     const __grid_constant__ CellScales sc,
                                                     const unsigned* pahabs, double eps, int pah0,
                                                     int n_pah, long long first, long long n,
                                                     float* X, float* p_abs, float* power,
                                                     const int* list) {
  const long long r0 = ((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5) * 32;
  const int lane = threadIdx.x & 31;
  const long long rows = n * n_pah;
  if (r0 >= rows) return;
  const int F = t.K + 2;
  // this lane's row
  const long long mine = r0 + lane < rows ? r0 + lane : rows - 1;
  const int p = pah0 + (int)(mine / n);
  const long long c = mine % n;
  const long long cell = first + (list ? (long long)list[c] : c);
  const float rho = g.rho[cell * g.S + t.species[p]];
  const long long at = (long long)p * g.n_leaves + cell;
  unsigned long long tot = 0;
  constexpr int kAhead = 4;  // rows in flight
  for (int i0 = 0; i0 < 32; i0 += kAhead) {
    unsigned c0[kAhead], c1[kAhead];
    bool dusty[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const unsigned* cnt = pahabs + (size_t)__shfl_sync(0xffffffffu, at, i0 + u) * t.K;
      dusty[u] = __shfl_sync(0xffffffffu, rho, i0 + u) > 0.0f;
      // K is at most 64: two bins a lane
      c0[u] = lane < t.K ? __ldg(&cnt[lane]) : 0u;
      c1[u] = lane + 32 < t.K ? __ldg(&cnt[lane + 32]) : 0u;
    }
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const unsigned long long sum =
          (unsigned long long)__reduce_add_sync(0xffffffffu, (c0[u] & 0xffffu) + (c1[u] & 0xffffu)) +
          ((unsigned long long)__reduce_add_sync(0xffffffffu, (c0[u] >> 16) + (c1[u] >> 16)) << 16);
      if (lane == i0 + u) tot = sum;
      if (r0 + i0 + u >= rows) continue;
      float* x = X + (size_t)(r0 + i0 + u) * F;
      // the shape features in FP32 (they enter a BF16 network)
      const bool on = sum != 0 && dusty[u];
      const float inv = on ? 1.0f / (float)sum : 0.0f;
      if (lane < t.K)
        x[lane] = on ? logf((float)c0[u] * inv + 1e-4f) * (1.0f / 4.6f) + 1.0f : 0.0f;
      if (lane + 32 < t.K)
        x[lane + 32] = on ? logf((float)c1[u] * inv + 1e-4f) * (1.0f / 4.6f) + 1.0f : 0.0f;
    }
  }
  if (r0 + lane >= rows) return;
  float xp = 0.0f, size = 0.0f, pa = 0.0f;
  if (tot != 0 && rho > 0.0f) {
    const double pw = (double)tot * eps;
    xp = (float)((log10(pw / ((double)rho * sc.molecules[p][g.level[cell]])) + 12.0) / 4.0);
    size = (float)sc.size_feature[p];
    pa = (float)pw;
  }
  float* x = X + (size_t)(r0 + lane) * F;
  x[t.K] = xp;
  x[t.K + 1] = size;
  p_abs[r0 + lane] = pa;
  if (power) power[r0 + lane] = xp;
}

// Training targets: y_b = ln(J_b / P_abs + 1e-6) / 7 + 1 from the exact emission (bins
// below 1e-6 of the cell's power carry no energy worth learning).
__global__ void k_pah_encode(const float* J, const float* p_abs, long long n, int B, float* Y) {
  long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (idx >= n * B) return;
  long long c = idx / B;
  float pa = p_abs[c];
  Y[idx] = pa > 0.0f ? logf(J[idx] / pa + 1e-6f) * (1.0f / 7.0f) + 1.0f : 0.0f;
}

// decoded surrogate output of one bin: q = max(exp(7 (y - 1)) - 1e-6, 0), FP32
__device__ __forceinline__ float decode_q(float y) {
  return fmaxf(expf(7.0f * (y - 1.0f)) - 1e-6f, 0.0f);
}

// The surrogate's emission of cells c < n: per PAH q_b = max(exp(7 (y_b - 1)) - 1e-6, 0)
// from row p n + c of Y, scaled to the absorbed power, summed over the PAHs into row list[c]
// (or c) of j_out. A PAH whose energy residual |sum_b q_b - 1| (before scaling) exceeds tol or
// whose power feature lies outside [x_lo, x_hi] flags the cell: it is appended to
// fallback[*n_fallback ..] (list[c], or off + c without a list), and with `leave` its row is
// left alone for the exact solution. n_fallback[1] becomes nonzero where the network's error
// word is (a wait of its pass ran out: Y is not to be used). One warp per cell; Y is read once,
// a lane's bins of every PAH in flight together. (Separate passes for the checks and for
// each PAH's sum, decoding twice and adding into j_out, took 170 us for 2.7e4 cells, two
// PAHs and 200 bins; this 32.)
constexpr int kFinishBins = 8;  // bins of a lane held in registers at a time

__global__ void k_surrogate_finish(const float* Y, const float* power, const float* p_abs,
                                   long long n, int n_pah, int B, float tol, float x_lo,
                                   float x_hi, bool leave, float* j_out, const int* list,
                                   int off, int* fallback, unsigned* n_fallback,
                                   const unsigned* net_err) {
  const long long c = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (c >= n) return;
  if (c == 0 && lane == 0 && *net_err) n_fallback[1] = 1u;
  float scale[kMaxPah];
  bool flagged = false;
#pragma unroll
  for (int p = 0; p < kMaxPah; ++p) {
    scale[p] = 0.0f;
    if (p >= n_pah) continue;
    const long long row = p * n + c;
    const float pa = p_abs[row];
    if (!(pa > 0.0f)) continue;
    float sum = 0.0f;
    for (int b0 = 0; b0 < B; b0 += 32 * kFinishBins) {
      float y[kFinishBins];
#pragma unroll
      for (int i = 0; i < kFinishBins; ++i) {
        const int b = b0 + 32 * i + lane;
        y[i] = b < B ? __ldg(&Y[row * B + b]) : -1e30f;
      }
#pragma unroll
      for (int i = 0; i < kFinishBins; ++i)
        if (b0 + 32 * i + lane < B) sum += decode_q(y[i]);
    }
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    const float xp = power[row];
    flagged |= !(fabsf(sum - 1.0f) <= tol) || xp < x_lo || xp > x_hi;
    if (sum > 0.0f) scale[p] = pa / sum;
  }
  if (flagged) {
    if (lane == 0) fallback[atomicAdd(n_fallback, 1u)] = list ? list[c] : off + (int)c;
    if (leave) return;
  }
  float* j = j_out + (size_t)(list ? (long long)list[c] : c) * B;
  for (int b0 = 0; b0 < B; b0 += 32 * kFinishBins) {
    float out[kFinishBins];
#pragma unroll
    for (int i = 0; i < kFinishBins; ++i) out[i] = 0.0f;
#pragma unroll
    for (int p = 0; p < kMaxPah; ++p) {
      if (!(scale[p] > 0.0f)) continue;
#pragma unroll
      for (int i = 0; i < kFinishBins; ++i) {
        const int b = b0 + 32 * i + lane;
        if (b < B) out[i] = fmaf(scale[p], decode_q(__ldg(&Y[(p * n + c) * B + b])), out[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < kFinishBins; ++i)
      if (b0 + 32 * i + lane < B) j[b0 + 32 * i + lane] = out[i];
  }
}

// Compaction: rows i < n whose cell first + i absorbed in a PAH (any, or only `pah`: the
// cell's flag word) are appended to out (order not kept); *count receives their number.
__global__ void k_compact(const unsigned* pah_flag, int pah, long long first, long long n,
                          int* out, unsigned* count) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const bool sel =
      i < n && (pah_flag[first + i] & (pah >= 0 ? 1u << pah : ~0u)) != 0u;
  const unsigned m = __ballot_sync(0xffffffffu, sel);
  if (!m) return;
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(m) - 1;
  unsigned base = 0;
  if (lane == leader) base = atomicAdd(count, (unsigned)__popc(m));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (sel) out[base + __popc(m & ((1u << lane) - 1u))] = (int)i;
}

// Zero the absorbed spectra of the PAH-active cells and their flags (the other
// rows are zero already). Each lane reads one cell's flag word (coalesced); the warp
// then clears the rows of its flagged cells one after another, a coalesced row of K
// words per PAH.
__global__ void k_pah_clear(const unsigned* pah_flag, long long N, int K, int n_pah,
                            unsigned* pahabs, unsigned* flag_out) {
  const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
  const int lane = threadIdx.x & 31;
  const long long w0 = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  for (long long base = w0 * 32; base < N; base += warps * 32) {
    const long long c = base + lane;
    const unsigned f = c < N ? pah_flag[c] : 0u;
    unsigned m = __ballot_sync(0xffffffffu, f != 0u);
    while (m) {
      const int src = __ffs(m) - 1;
      m &= m - 1;
      const unsigned fc = __shfl_sync(0xffffffffu, f, src);
      const long long cc = base + src;
      for (int p = 0; p < n_pah; ++p)
        if (fc & (1u << p))
          for (int k = lane; k < K; k += 32) pahabs[((size_t)p * N + cc) * K + k] = 0u;
    }
    if (f) flag_out[c] = 0u;
  }
}

}  // namespace

cudaError_t launch_pah_tables(const PahBuild& pb, const PahTables& t, cudaStream_t s) {
  int n = pb.n_pah * pb.M;
  k_pah_temps<<<(n + 31) / 32, 32, 0, s>>>(pb);
  k_pah_levels<<<(n + 3) / 4, 128, 0, s>>>(pb);
  int nk = pb.n_pah * pb.K;
  k_pah_coarse<<<(nk + 63) / 64, 64, 0, s>>>(pb);
  const int nf = pb.n_pah * (pb.M + 1) > nk ? pb.n_pah * (pb.M + 1) : nk;
  k_pah_f32<<<(nf + 63) / 64, 64, 0, s>>>(pb);
  size_t smem = sizeof(double) * (t.K + 2 * t.M);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k_pah_template,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  k_pah_template<<<pb.n_pah, 32, smem, s>>>(t, pb);
  return cudaGetLastError();
}

static CellScales cell_scales(const PahTables& t, double eps, double d0) {
  CellScales sc{};
  for (int p = 0; p < t.n_pah; ++p) {
    for (int l = 0; l < kMaxLevels; ++l) {
      const double V = d0 * d0 * d0 / (double)(1ll << (3 * l));
      sc.molecules[p][l] = V / (d0 * t.mol_mass[p]);
      sc.eps_per_molecule[p][l] = eps / sc.molecules[p][l];
    }
    sc.size_feature[p] = log10((double)t.n_carbon[p]) - 2.0;
  }
  return sc;
}

template <int kMinBlocks>
static cudaError_t launch_exact_variant(const DevGrid& g, const PahTables& t,
                                        const CellScales& sc, const unsigned* pahabs,
                                        long long first, long long n, float* j_out, int pah_only,
                                        cudaStream_t s, const int* list, const int* cell_of_row) {
  const size_t smem = sizeof(float) * (size_t)exact_cell_floats(t.M) * kCells;
  cudaError_t e = cudaFuncSetAttribute(k_pah_exact<kMinBlocks>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_pah_exact<kMinBlocks><<<(unsigned)((n + kCells - 1) / kCells), 8 * kCells, smem, s>>>(
      g, t, sc, pahabs, first, n, j_out, pah_only, list, cell_of_row);
  return cudaGetLastError();
}

// Eight cells a block: a block's barriers between solving and forming the emission hold up
// few warps, and the level table comes from L1 and L2 often enough (5.0e4 cells with all
// else equal: 32 cells a block 1.41 ms a call, 16 1.40, 8 1.32). Eight blocks an SM (128
// registers) where there are that many; with fewer cells the registers of four (1.0e3
// cells: 0.15 against 0.21 ms).
cudaError_t launch_pah_exact(const DevGrid& g, const PahTables& t, const unsigned* pahabs,
                             double eps, double d0, long long first, long long n,
                             float* j_out, int pah_only, cudaStream_t s, const int* list,
                             const int* cell_of_row) {
  if (n <= 0) return cudaSuccess;
  const CellScales sc = cell_scales(t, eps, d0);
  const size_t per_cell = sizeof(float) * (size_t)exact_cell_floats(t.M);
  if (per_cell * kCells > 220 * 1024) return cudaErrorInvalidValue;
  if (n > 4ll * kCells * 152)
    return launch_exact_variant<8>(g, t, sc, pahabs, first, n, j_out, pah_only, s, list,
                                   cell_of_row);
  return launch_exact_variant<4>(g, t, sc, pahabs, first, n, j_out, pah_only, s, list,
                                 cell_of_row);
}

}  // namespace rt

namespace rt {

cudaError_t launch_pah_features(const DevGrid& g, const PahTables& t, const unsigned* pahabs,
                                double eps, double d0, int pah0, int n_pah, long long first,
                                long long n, float* X, float* p_abs, float* power,
                                cudaStream_t s, const int* list) {
  if (n <= 0) return cudaSuccess;
  k_pah_features<<<(unsigned)((n * n_pah + 63) / 64), 64, 0, s>>>(
      g, t, cell_scales(t, eps, d0), pahabs, eps, pah0, n_pah, first, n, X, p_abs, power, list);
  return cudaGetLastError();
}

cudaError_t launch_pah_encode(const float* J, const float* p_abs, long long n, int B, float* Y,
                              cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  long long m = n * B;
  k_pah_encode<<<(unsigned)((m + 255) / 256), 256, 0, s>>>(J, p_abs, n, B, Y);
  return cudaGetLastError();
}

cudaError_t launch_surrogate_finish(const float* Y, const float* power, const float* p_abs,
                                    long long n, int n_pah, int B, float tol, float x_lo,
                                    float x_hi, bool leave, float* j_out, const int* list,
                                    int off, int* fallback, unsigned* n_fallback,
                                    const unsigned* net_err, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_surrogate_finish<<<(unsigned)((n + 3) / 4), 128, 0, s>>>(Y, power, p_abs, n, n_pah, B, tol,
                                                             x_lo, x_hi, leave, j_out, list, off,
                                                             fallback, n_fallback, net_err);
  return cudaGetLastError();
}

// P(T) of a PAH in a monochromatic field (Fig. 3): levels E_f = f dE up to E(t_top) +
// h nu. Four kernels over all cases of a call: the level temperatures (a thread per
// level), the levels' emission per bin and cooling rates (a warp per level; FP64-bound,
// so every bin edge is evaluated once and the spectra are kept for the last kernel), the
// populations by the level-by-level flux balance for the single photon energy (a warp
// per case, the recursion in one lane), the emission (a block per case and 32 bins).
// One block per case doing all of it, with every Planck integral twice, took 187 ms for
// 12 cases of 400 levels and 200 bins; the four kernels take 0.03 + 0.17 + 0.17 + 0.02
// ms, the call 0.61 ms with its copies and allocation.
__global__ void k_pt_temps(const PtCase* cases, int n_cases, int M, double* dE_out,
                           double* T_out) {
  const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (idx >= (long long)n_cases * M) return;
  const int c = (int)(idx / M), f = (int)(idx % M);
  const PtCase& cs = cases[c];
  const double dE = (heat_content(cs.t_top, cs.spec) + cs.h_nu) / (double)(M - 1);
  if (f == 0) dE_out[c] = dE;
  T_out[idx] = f == 0 ? 0.0 : level_temperature(f * dE, cs.spec);
}

__global__ void k_pt_levels(int n_cases, const double* nu, int B, const double* sigma, int M,
                            const double* dE, const double* T, double* spec, double* cool) {
  const long long idx = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  if (idx >= (long long)n_cases * M) return;
  const int c = (int)(idx / M);
  const double* sig = sigma + (size_t)c * B;
  double* s = spec + (size_t)idx * B;
  double L = 0.0;
  planck::planck_bins_warp(nu, B, T[idx], [&](int b, double v) {
    v *= sig[b];
    s[b] = v;
    L += v;
  });
  for (int o = 16; o > 0; o >>= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
  if ((threadIdx.x & 31) == 0) cool[idx] = 4.0 * kPi * L / dE[c];  // steps down per second
}

// The flux F up across the boundary below level f equals cooling across it, P_f = F / C_f;
// then F changes by what leaves level f upwards less what has arrived there: from level
// f - q (weight 1 - w) and f - q - 1 (weight w), one photon being q + w levels. A serial
// chain over the levels in one lane: the reciprocals of C are formed in parallel before
// it, so a step is one product, one fused multiply-add and a maximum deep (with the
// division and the arrivals scattered through shared memory a step took 1.0 us, now 0.4).
// Shared memory: P and 1/C, M doubles each.
__global__ void __launch_bounds__(32) k_pt_populations(const PtCase* cases, int M,
                                                       const double* dE, const double* cool,
                                                       const double* T, double t_sub,
                                                       double* P_out, double* p_above) {
  extern __shared__ double sm[];
  double* P = sm;
  double* rC = P + M;
  const PtCase& c = cases[blockIdx.x];
  const int lane = threadIdx.x;
  const size_t row = (size_t)blockIdx.x * M;
  for (int f = lane; f < M; f += 32) {
    const double C = cool[row + f];
    rC[f] = C > 0.0 ? fmin(1.0 / C, 1e308) : 0.0;
  }
  __syncwarp();
  if (lane == 0) {
    const double x = c.h_nu / dE[blockIdx.x];
    const int q = (int)floor(x);
    const double w = x - floor(x);
    const double r0 = q > 0 ? c.rate * (1.0 - w) : 0.0, r1 = c.rate * w;
    // upward rate out of level i; absorptions beyond the top level end there
    auto up = [&](int i) { return i + q < M - 1 ? r0 + r1 : (i < M - 1 ? c.rate : 0.0); };
    P[0] = 1.0;
    double F = up(0);
    for (int f = 1; f < M; ++f) {
      const double D = (f > q ? r1 * P[f - q - 1] : 0.0) + (q > 0 && f >= q ? r0 * P[f - q] : 0.0);
      const double Pf = F * rC[f];
      P[f] = Pf;
      F = fmax(fma(Pf, up(f), F - D), 0.0);
      if (Pf > 1e250) {  // keep the numbers finite
        for (int i = 0; i <= f; ++i) P[i] *= 1e-250;
        F *= 1e-250;
      }
    }
  }
  __syncwarp();
  double tot = 0.0, a = 0.0;
  for (int f = lane; f < M; f += 32) tot += P[f];
  for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
  for (int f = lane; f < M; f += 32) {
    const double v = P[f] / tot;
    P_out[row + f] = v;
    if (T[row + f] > t_sub) a += v;
  }
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  if (lane == 0) p_above[blockIdx.x] = a;
}

constexpr int kPtWarps = 8;

__global__ void __launch_bounds__(32 * kPtWarps) k_pt_emission(int B, int M, const double* spec,
                                                               const double* P, double* em_out) {
  __shared__ double part[kPtWarps][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = blockIdx.y * 32 + lane;
  const size_t row = (size_t)blockIdx.x * M;
  double e = 0.0;
  if (b < B)
    for (int f = warp; f < M; f += kPtWarps) e += P[row + f] * spec[(row + f) * B + b];
  part[warp][lane] = e;
  __syncthreads();
  if (warp == 0 && b < B) {
    for (int i = 1; i < kPtWarps; ++i) e += part[i][lane];
    em_out[(size_t)blockIdx.x * B + b] = 4.0 * kPi * e;
  }
}

size_t pt_scratch_doubles(int n_cases, int M, int B) {
  return (size_t)n_cases * (1 + M + (size_t)M * B);
}

// scratch: pt_scratch_doubles(n_cases, M, B) doubles
cudaError_t launch_pah_pt(const PtCase* cases, int n_cases, const double* nu, int B,
                          const double* sigma, int M, double t_sub, double* P_out,
                          double* T_out, double* p_above, double* em_out, double* scratch,
                          cudaStream_t s) {
  double* dE = scratch;
  double* cool = dE + n_cases;
  double* spec = cool + (size_t)n_cases * M;
  const size_t smem = sizeof(double) * 2 * (size_t)M;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(
        k_pt_populations, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  const long long n = (long long)n_cases * M;
  k_pt_temps<<<(unsigned)((n + 31) / 32), 32, 0, s>>>(cases, n_cases, M, dE, T_out);
  k_pt_levels<<<(unsigned)((n + 3) / 4), 128, 0, s>>>(n_cases, nu, B, sigma, M, dE, T_out, spec,
                                                      cool);
  k_pt_populations<<<n_cases, 32, smem, s>>>(cases, M, dE, cool, T_out, t_sub, P_out, p_above);
  k_pt_emission<<<dim3(n_cases, (B + 31) / 32), 32 * kPtWarps, 0, s>>>(B, M, spec, P_out, em_out);
  return cudaGetLastError();
}

// Per-cell re-emission spectra: each row of J [n][B] (erg/s per bin; negative or NaN
// entries count as 0) becomes its normalised cumulative sum, the last entry exactly
// 1; a row with nothing positive becomes zeros (the transport then uses the
// template). One warp per row, FP64 sums, a 32-wide inclusive scan per chunk.
__global__ void k_pah_cell_cdf(const float* J, long long n, int B, float* out) {
  const int lane = threadIdx.x & 31;
  const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
  for (long long row = blockIdx.x * (long long)(blockDim.x >> 5) + (threadIdx.x >> 5); row < n;
       row += warps) {
    const float* j = J + row * B;
    float* o = out + row * B;
    double tot = 0.0;
    for (int b = lane; b < B; b += 32) tot += (double)fmaxf(j[b], 0.f);
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, s);
    if (!(tot > 0.0)) {
      for (int b = lane; b < B; b += 32) o[b] = 0.f;
      continue;
    }
    double carry = 0.0;
    for (int base = 0; base < B; base += 32) {
      const int b = base + lane;
      double v = b < B ? (double)fmaxf(j[b], 0.f) : 0.0;
#pragma unroll
      for (int s = 1; s < 32; s <<= 1) {
        const double u = __shfl_up_sync(0xffffffffu, v, s);
        if (lane >= s) v += u;
      }
      if (b < B) o[b] = b == B - 1 ? 1.f : (float)((carry + v) / tot);
      carry += __shfl_sync(0xffffffffu, v, 31);
    }
  }
}

cudaError_t launch_pah_cell_cdf(const float* J, long long n, int B, float* out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  long long blocks = (n + 7) / 8;
  if (blocks > 65536) blocks = 65536;
  k_pah_cell_cdf<<<(unsigned)blocks, 256, 0, s>>>(J, n, B, out);
  return cudaGetLastError();
}

cudaError_t launch_compact(const unsigned* pah_flag, int pah, long long first, long long n,
                           int* out, unsigned* count, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_compact<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(pah_flag, pah, first, n, out, count);
  return cudaGetLastError();
}

cudaError_t launch_pah_clear(const unsigned* pah_flag, long long N, int K, int n_pah,
                             unsigned* pahabs, unsigned* flag_out, cudaStream_t s) {
  if (N <= 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  long long blocks = (N + 255) / 256;  // a lane per cell
  const long long cap = (long long)(sms > 0 ? sms : 152) * 8;
  if (blocks > cap) blocks = cap;
  k_pah_clear<<<(unsigned)blocks, 256, 0, s>>>(pah_flag, N, K, n_pah, pahabs, flag_out);
  return cudaGetLastError();
}

}  // namespace rt
