// rt_internal.h -- structures shared by the host side and the kernels of
// librt_gb300. Not part of the public ABI (include/rt.h is).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

struct rt_mlp;  // the network (rt_mlp.cu)

namespace rt {

constexpr int kMaxSpecies = 8;
constexpr int kMaxLevels = 8;     // levels 0 .. 7
constexpr int kMaxBins = 1024;
constexpr int kMaxPah = 4;        // PAH species per grid
constexpr int kMaxModeGroups = 4; // vibrational mode groups per PAH

// Device status bits.
constexpr unsigned kStatusTree = 1u;     // a package met a malformed tree
constexpr unsigned kStatusTimeout = 2u;  // a launch ran past its time budget

// Indices into the device counter array.
enum Counter {
  kCEmitted = 0, kCEscaped, kCCapped, kCAbsorptions, kCScatters, kCCrossings,
  kCErrors, kCClamped, kCLevels, kCPeelEvents, kCPeelCrossings, kCPeelDropped, kNumCounters
};

// Face links of a leaf (record of 8 int32 per leaf: faces -x,+x,-y,+y,-z,+z, then
// the densities of species 0 and 1 as float bits when S <= 2). A link is
//   kLinkEscape                the face is the domain boundary;
//   id | (levels up << 28)     the neighbouring leaf: 0 levels up a leaf of the same size
//                              (so links below kLinkSame need no decoding), else coarser;
//   -(block + 1)               the same-size neighbour is split: descend into block.
constexpr int32_t kLinkEscape = (int32_t)0x80000000;
constexpr int32_t kLinkLeafMask = 0x0FFFFFFF;
constexpr int32_t kLinkSame = 1 << 28;
constexpr long long kMaxLinkedLeaves = 1ll << 28;

// Path-length tallies lie species by species within a cell, in rows of this many floats: whole
// vectors for the reductions (see tally_segment).
__host__ __device__ constexpr int tally_row(int S) { return S <= 2 ? S : (S + 3) & ~3; }

// The row of a leaf: within blocks of 4096 leaves the two 6-bit halves of the number trade
// places (which undoes itself), so that cells close together lie 64 rows apart. Reductions to one
// memory line are done one after another, and leaves are numbered along a space-filling curve:
// in order, the cells that every package crosses next to the source share a few lines, and the
// time of a launch went by which parts of L2 those lines fell into. 2e6 packages through 1.06e6
// cells of two species, the array moved by 0 to 32 MB: 2.28 to 3.25 ms in order, 1.90 to 1.98 so
// (blocks of 1024 1.97 to 2.10, of 16384 1.91 to 2.06); 4e6 through 1.9e7 cells 16.5 and 14.4;
// 1e6 through 5.9e4 1.83 and 0.85.
constexpr int kTallyBits = 6;
constexpr long long kTallyBlock = 1ll << (2 * kTallyBits);
__host__ __device__ constexpr size_t tally_place(long long leaf) {
  constexpr long long m = (1ll << kTallyBits) - 1;
  return (size_t)((leaf & ~(kTallyBlock - 1)) | (leaf & m) << kTallyBits | (leaf >> kTallyBits & m));
}
__host__ __device__ constexpr size_t tally_floats(int S, long long n_leaves) {
  return (size_t)((n_leaves + kTallyBlock - 1) / kTallyBlock * kTallyBlock) * tally_row(S);
}

// Geometry and densities (device pointers), passed by value.
struct DevGrid {
  const int32_t* base;     // [n^3]
  const int32_t* child;    // [n_blocks*8]
  const float* rho;        // [n_leaves][S]: density times the base-cube edge, g cm^-2
  const int8_t* level;     // [n_leaves] refinement level of every leaf
  const int32_t* links;    // [n_leaves][8] face links (+ densities when S <= 2)
  // densities by tree slot for the path walk: [n_base^3 + 8 n_blocks][S], slot i < n^3
  // the base cell i, slot n^3 + 8 b + o the child o of block b; zeros where refined
  const float* rho_slot;
  long long n_leaves, n_blocks;
  int n_base, max_level, S, B, n_dir, n_T;
  int n_base3;             // n_base^3, the first block slot
};

// Face-link record of a leaf, 8 words (32 bytes): links of faces -x,+x,-y,+y,-z,+z,
// then the densities of species 0 and 1 when S <= 2 (zero otherwise).
constexpr int kRec = 8;

// Per-bin opacity record for one species.
struct alignas(16) Kappa {
  float kext, ksca, kabs, g;  // cm^2 g^-1, cm^2 g^-1, cm^2 g^-1, HG asymmetry
};

// Tables built in FP64 on the device and stored for transport.
struct DevTables {
  const Kappa* kap;           // [B][S]
  const float* kext;          // [B][S] the records' extinction opacities alone
  const float* star_cdf;      // [B] normalised cumulative stellar spectrum
  const float* S32;           // [S][n_T] emitted power per gram at the table rows
  const double* S64;          // [S][n_T]
  const double* Tgrid;        // [n_T], Tgrid[0] = 0
  const float* dcdf;          // [S][n_T-1][B] normalised cumulative of row differences
  const unsigned short* cdf_guide;  // [S][n_T-1][B]: first bin whose cdf exceeds k/B
  const int* u_guide;         // [S][n_T]: interval holding exp(u_ln0 + k / u_inv)
  float u_ln0[kMaxSpecies];   // ln S_s(T_1)
  float u_inv[kMaxSpecies];   // (n_T - 1) / (ln S_s(T_last) - ln S_s(T_1))
  const float* u_frozen;      // [S][n_leaves] (frozen mode) or null
  const float* pah_cdf;       // [n_pah][B] template re-emission spectrum of each PAH
  const float* pah_cell_cdf;  // [n_pah][n_leaves][B] per-cell PAH re-emission spectra
                              // (normalised cumulative; last entry 0: the template), or null
  int pah_of[kMaxSpecies];    // PAH number of each species, -1 for grains
  int n_coarse;               // coarse bins of the PAH absorbed spectrum
  float u_tmin[kMaxSpecies];  // S_s(t_min)
  float eps_d0_over_V[kMaxLevels];   // eps * d0 / V(level), erg s^-1 cm^-2 (FP32)
  double eps_over_V[kMaxLevels];     // eps / V(level) (FP64, temperatures)
  double d0;                  // base-cube edge, cm
};

// One transport launch.
struct DevRun {
  unsigned long long seed, first_id, n_packages, max_events;
  unsigned long long* next;       // pool: packages handed out so far
  unsigned long long* count;      // [S][n_leaves]
  unsigned long long* sed;        // [2][n_dir][B]
  unsigned long long* counters;   // [kNumCounters]
  unsigned int* status;
  unsigned* pahabs;               // [n_pah][n_leaves][n_coarse] PAH absorptions
  unsigned* pah_flag;             // [n_leaves] bit p set: PAH p absorbed in the cell
  float* pathabs;                 // path-length tallies, rows tally_place(leaf), or null
  float src[3];                   // source position, base-cube units
  float beam[3];
  double src64[3];
  double beam64[3];
  int source_kind, mode, refill_period;
  int interaction_batch;          // pool: waiting lanes that trigger an interaction phase
  float count_scale;              // BW / no-correction: temperature index = scale x count
  int sed_in_smem;                // pool: escaped-spectrum histogram in shared memory
  unsigned long long budget_ns;
};

// Peel-off images toward a distant observer. Every scattering and re-emission at a
// bin that has an image plane sends the share w of the package's energy per
// steradian toward the observer (HG phase function value, or 1/(4 pi)), attenuated
// by exp(-tau) along the sight line to the boundary, into the pixel its position
// projects to. The transport launch only records these events (position, w, bin);
// a second kernel traces their sight lines. Emissions by a point source are counted
// per bin and peeled once per bin after the launch (they all start at the source).
struct DevPeel {
  const int* plane_of_bin;       // [B] image plane of each bin, -1 for none
  double* image;                 // [n_planes][ny][nx] sums of w exp(-tau) (times eps: erg/s/sr)
  unsigned long long* n_emit;    // [B] point-source emissions since the last source peel
  float4* ev;                    // [capacity] recorded events: position (base units), w
  int* ev_bin;                   // [capacity] their bins
  unsigned long long* n_ev;      // events recorded by the current launch
  unsigned long long capacity;
  float o[3];                    // unit vector toward the observer
  float e1[3], e2[3];            // image axes: e1 = normalise(z x o) (x when o ~ z), e2 = o x e1
  float centre;                  // model centre, base-cube units
  float sx, sy;                  // pixels per base-cube unit along e1, e2
  int nx, ny, n_planes;
  float tau_max;                 // sight lines stop (contribute nothing) beyond this depth
};

constexpr int kMaxImageSide = 16384;
constexpr unsigned long long kPeelCapacityDefault = 1ull << 24;
constexpr unsigned long long kPeelCapacityMax = 1ull << 31;
constexpr size_t kMaxImagePixels = (size_t)1 << 28;  // all planes together (2 GiB of FP64)

// One model of a batched launch.
struct ModelDesc {
  DevGrid g;
  DevTables t;
  DevRun r;
  float* T_out;  // temperatures [S][n_leaves] of the model
};

// The packages of a batched launch.
struct BatchQueue {
  const unsigned long long* plan;    // [n] of each model
  const unsigned long long* before;  // [n + 1] of the models before it
  unsigned long long* next;          // [n] of each model handed out so far, then the number of
                                     // models found exhausted (zeros at the start)
  int n, n_live;                     // models, and those with packages
};
constexpr unsigned long long kExhausted = 1ull << 63;  // set in next[m] by the first to find it so

// Kernel launchers (rt_transport.cu, rt_tables.cu).
// chunk >= 32: how many packages a warp takes at a time. s_fixed: the species count all
// models share (2 has a walk compiled for it), 0 otherwise; tally: the path-length tallies
// (of every model)
cudaError_t launch_transport_batch(const ModelDesc* models, const BatchQueue& q, int chunk,
                                   int blocks_per_sm, int s_fixed, bool tally, int threads,
                                   cudaStream_t s);
cudaError_t launch_transport_pool(const DevGrid& g, const DevTables& t, const DevRun& r,
                                  int blocks_per_sm, int threads, cudaStream_t s,
                                  const DevPeel* peel = nullptr, bool path = false);
cudaError_t launch_peel_source(const DevGrid& g, const DevTables& t, const DevRun& r,
                               const DevPeel& peel, cudaStream_t s);
cudaError_t launch_peel_trace(const DevGrid& g, const DevTables& t, const DevRun& r,
                              const DevPeel& peel, cudaStream_t s);
cudaError_t launch_image_out(const double* image, long long n, double scale, double* out,
                             cudaStream_t s);
cudaError_t launch_image_profile(const double* image, int nx, int ny, int plane_a,
                                 int plane_b, int half_rows, double scale, double* out,
                                 cudaStream_t s);
cudaError_t launch_transport_plain(const DevGrid& g, const DevTables& t, const DevRun& r,
                                   bool fp64, int threads, cudaStream_t s);
// One event of a replayed history (rt_trace_events): kind 0 emission, 1 scattering,
// 2 absorption, 3 escape, 4 capped; position in base-cube units.
struct TraceEvent {
  int kind, species, leaf, bin;
  float pos[3];
  int pad;
};
cudaError_t launch_trace(const DevGrid& g, const DevTables& t, const DevRun& r,
                         const unsigned long long* ids, long long n, long long* out,
                         cudaStream_t s, TraceEvent* ev = nullptr, long long ev_cap = 0,
                         long long* ev_n = nullptr);
cudaError_t launch_build_links(const DevGrid& g, const int32_t* leaf_ijk, int32_t* links,
                               cudaStream_t s);
cudaError_t launch_build_rho_slot(const DevGrid& g, float* rho_slot, cudaStream_t s);

// Device walk of the tree (rt_grid.cu): inputs, outputs and work arrays.
struct TreeBuild {
  const int32_t* base;     // [n^3]
  const int32_t* child;    // [n_blocks][8]
  long long n_leaves, n_blocks;
  int n_base, max_level;
  int8_t* level;           // [n_leaves] out
  int32_t* ijk;            // [n_leaves][3] out: integer corner at the leaf's level
  int8_t* blk_level;       // [n_blocks] work
  int32_t* blk_ijk;        // [n_blocks][3] work
  unsigned* leaf_seen;     // [(n_leaves + 31) / 32] work bitmap
  unsigned* blk_seen;      // [(n_blocks + 31) / 32] work bitmap
  unsigned* err;           // nonzero: malformed tree (bit 0) or bad density (bit 1)
  int* max_seen;           // deepest level reached
};
cudaError_t launch_tree_walk(const TreeBuild& tb, cudaStream_t s);
cudaError_t launch_rho_convert(const double* src, long long N, int S, double d0, float* dst,
                               unsigned* err, cudaStream_t s);
cudaError_t launch_philox(const unsigned long long* ids, long long n, unsigned event,
                          unsigned block, unsigned long long seed, unsigned* out,
                          cudaStream_t s);

struct TableBuild {
  int S, B, n_T;
  const double* nu;          // [B+1]
  const double* kabs;        // [S][B]
  const double* ksca;        // [S][B]
  const double* ghg;         // [S][B]
  double T_star, t_min, t_max;
  // outputs
  double* Tgrid;             // [n_T]
  double* P;                 // scratch [n_T][B]
  double* S64;               // [S][n_T]
  float* S32;                // [S][n_T]
  float* dcdf;               // [S][n_T-1][B]
  unsigned short* cdf_guide; // [S][n_T-1][B]
  int* u_guide;              // [S][n_T]
  Kappa* kap;                // [B][S]
  float* kext;               // [B][S]
  float* star_cdf;           // [B]
  double* star_frac;         // [1] in-range fraction of the stellar blackbody
};
cudaError_t launch_build_tables(const TableBuild& tb, cudaStream_t s);

// PAH molecular data: vibrational mode groups (count, characteristic temperature)
struct PahSpec {
  int n_groups;
  double n_modes[kMaxModeGroups];
  double theta[kMaxModeGroups];
};

struct PahBuild {
  int n_pah, M, K, B;
  const double* nu;          // [B+1]
  const double* sigma;       // [n_pah][B] cross section per molecule, cm^2
  PahSpec spec[kMaxPah];
  double dE[kMaxPah];        // level spacing, erg
  double T_star, f_ref;      // template heating: source blackbody at bolometric flux f_ref
  float* s;                  // [n_pah][M/2][B][2] emission per level and bin, erg/s (M and
                             // B padded to multiples of 4)
  double* L;                 // [n_pah][M] cooling rate per level, erg/s
  double* T;                 // [n_pah][M] level temperatures (work array)
  double* e_k;               // [K] photon energy of each coarse bin, erg
  int* q_k;                  // [n_pah][K] floor(e_k / dE)
  double* w_k;               // [n_pah][K] e_k / dE - q_k
  float* template_cdf;       // [n_pah][B]
  float* c_f;                // [n_pah][M] downward rate L_f / dE, 1/s (FP32 copy)
  float* w_f;                // [n_pah][K] w_k (FP32 copy)
  float* e_f;                // [K] e_k (FP32 copy)
  unsigned char* first_k;    // [n_pah][M + 1] coarse bins with q_k < d
};

struct PahTables {
  int n_pah, M, K;
  const float* s;
  const double* L;
  const double* e_k;
  const int* q_k;
  const double* w_k;
  const float* c_f;          // [n_pah][M] L_f / dE in FP32
  const float* w_f;          // [n_pah][K] w_k in FP32
  const float* e_f;          // [K] e_k in FP32
  const unsigned char* first_k;  // [n_pah][M + 1] coarse bins with q_k < d
  double dE[kMaxPah];
  double mol_mass[kMaxPah];  // g per molecule
  int species[kMaxPah];      // species index of each PAH
  int n_carbon[kMaxPah];     // C atoms of each PAH
};

cudaError_t launch_pah_tables(const PahBuild& pb, const PahTables& t, cudaStream_t s);
cudaError_t launch_pah_exact(const DevGrid& g, const PahTables& t, const unsigned* pahabs,
                             double eps, double d0, long long first, long long n,
                             float* j_out, int pah_only, cudaStream_t s,
                             const int* list = nullptr, const int* cell_of_row = nullptr);
cudaError_t launch_pah_features(const DevGrid& g, const PahTables& t, const unsigned* pahabs,
                                double eps, double d0, int pah0, int n_pah, long long first,
                                long long n, float* X, float* p_abs, float* power,
                                cudaStream_t s, const int* list = nullptr);
cudaError_t launch_pah_encode(const float* J, const float* p_abs, long long n, int B, float* Y,
                              cudaStream_t s);
cudaError_t launch_surrogate_finish(const float* Y, const float* power, const float* p_abs,
                                    long long n, int n_pah, int B, float tol, float x_lo,
                                    float x_hi, bool leave, float* j_out, const int* list,
                                    int off, int* fallback, unsigned* n_fallback,
                                    const unsigned* net_err, cudaStream_t s);
cudaError_t launch_pah_clear(const unsigned* pah_flag, long long N, int K, int n_pah,
                             unsigned* pahabs, unsigned* pah_flag_out, cudaStream_t s);
cudaError_t launch_compact(const unsigned* pah_flag, int pah, long long first, long long n,
                           int* out, unsigned* count, cudaStream_t s);
cudaError_t launch_pah_cell_cdf(const float* J, long long n, int B, float* out, cudaStream_t s);

// The network's device word that a wait that ran out sets.
const unsigned* mlp_error_word(const rt_mlp* m);

// One P(T) problem: a PAH in a monochromatic field.
struct PtCase {
  PahSpec spec;
  double h_nu;   // photon energy, erg
  double rate;   // absorbed photons per molecule per second
  double t_top;  // levels span 0 .. E(t_top) + h_nu
};
cudaError_t launch_pah_pt(const PtCase* cases, int n_cases, const double* nu, int B,
                          const double* sigma, int M, double t_sub, double* P_out,
                          double* T_out, double* p_above, double* em_out, double* scratch,
                          cudaStream_t s);
size_t pt_scratch_doubles(int n_cases, int M, int B);

cudaError_t launch_frozen_u(const DevGrid& g, const DevTables& t, const float* T_frozen,
                            float* u_frozen, float t_min, float t_max, cudaStream_t s);
// out [S][n_leaves] from tallies in rows tally_place(leaf)
cudaError_t launch_tally_out(const DevGrid& g, const float* pathabs, float* out, cudaStream_t s);
// Every model of a batch in one launch (max_cells: of the largest): temperatures from the
// counts into T_out; counts, spectra, counters and status to zero.
cudaError_t launch_batch_temperatures(const ModelDesc* models, int n_models, long long max_cells,
                                      int s_fixed, cudaStream_t s);
cudaError_t launch_batch_reset(const ModelDesc* models, int n_models, long long max_cells,
                               cudaStream_t s);
cudaError_t launch_temperatures(const DevGrid& g, const DevTables& t,
                                const unsigned long long* count, float* T_out,
                                unsigned long long* counters, cudaStream_t s,
                                const float* pathabs = nullptr);

}  // namespace rt
