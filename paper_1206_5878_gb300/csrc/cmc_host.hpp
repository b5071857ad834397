// Host-side internals of the CUDA library: the segment (cluster) layout on
// the device, scratch buffers, and the launchers of each kernel.  Nothing
// here is part of the C ABI (see include/cmc.h).
#pragma once

#include <cstdint>
#include <cstddef>
#include <string>
#include <utility>
#include <vector>

#include <cuda_runtime.h>

#include "cmc_device.cuh"

namespace cmc {

// Launch a kernel that calls pdl_enter: it may be set up while its
// predecessor in the stream still runs (in a captured graph the edge becomes
// a programmatic one).  An error is left for cudaGetLastError.
template <class... P, class... A>
inline void launch_k(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem,
                            cudaStream_t st, A&&... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

// Several device arrays in one stream-ordered allocation: first those with initial
// values (put), then zeroed ones (zero), then the rest (add).  A stage call on
// 10^6 stars spent more time on its 14 to 50 allocations, copies and fills (two
// to five microseconds of host work each) than on its kernels.  A small image
// goes as a kernel's argument, which the launch copies; a large one is copied
// from the host and waited for.
class Carve {
 public:
  template <class T>
  void put(T*& p, const T* src, size_t count) {
    const size_t at = claim((void**)&p, sizeof(T) * count, 32);
    image_.resize(bytes_, 0);
    if (count) copy(image_.data() + at, src, sizeof(T) * count);
    zero_ = bytes_;
  }
  template <class T>
  void zero(T*& p, size_t count) {
    claim((void**)&p, sizeof(T) * count, 32);
    zero_ = bytes_;
  }
  template <class T>
  void add(T*& p, size_t count) {
    claim((void**)&p, sizeof(T) * (count ? count : 1), 256);
  }
  cudaError_t alloc(void*& block, cudaStream_t st);

 private:
  struct Part {
    void** ptr;
    size_t at;
  };
  std::vector<Part> parts_;
  std::vector<unsigned char> image_;
  size_t bytes_ = 0, zero_ = 0;  // zero_: end of the zeroed part
  static void copy(unsigned char* to, const void* from, size_t n);
  size_t claim(void** p, size_t n, size_t align) {
    const size_t at = (bytes_ + align - 1) / align * align;
    parts_.push_back({p, at});
    bytes_ = at + (n + 31) / 32 * 32;
    return at;
  }
};

// Device-resident description of the segments of one state.  Offsets are
// fixed at initialisation; nb, dt and the statistics change every step.
struct SegLayout {
  int n_seg = 0;
  int64_t n = 0;          // total stars
  int64_t n_tiles = 0;    // tiles of kTile elements, never straddling segments
  int64_t n_pairs = 0;    // pair slots (floor(n_c / 2) summed)
  int64_t n_bins = 0;     // bin slots (ceil(n_c / bin_size) summed)
  int bin_size = 20;
  std::vector<int64_t> h_off, h_tile_off, h_pair_off, h_bin_off;
  int64_t max_seg = 0;    // stars of the largest segment
  // device arrays, all in one block
  void* block = nullptr;
  int64_t* off = nullptr;
  int64_t* tile_off = nullptr;
  int64_t* pair_off = nullptr;
  int64_t* bin_off = nullptr;
  uint64_t* seed = nullptr;
  double* lnL = nullptr;
  int64_t* nb = nullptr;
  int64_t* esc_step = nullptr;      // stars escaped during the current step
  uint64_t* dt_bits = nullptr;
  uint64_t* dt_last = nullptr;      // timestep of the last completed step
  double* dt_cap = nullptr;         // outside bounds on the timestep (cmc_set_dt_cap; 0: none)
  unsigned long long* stats = nullptr;
  double* esc_me = nullptr;         // [n_seg][2]: mass, energy carried off by escapers
  uint32_t* tile_done = nullptr;    // blocks of a tile that have finished; zero between kernels
  uint4* taus = nullptr;            // combined-Tausworthe streams (stream mode only)
  int64_t* taus_base = nullptr;     // per segment: first stream slot
  int64_t taus_slots = 0;

  Seg dev() const {
    Seg s;
    s.off = off; s.tile_off = tile_off; s.pair_off = pair_off; s.bin_off = bin_off;
    s.seed = seed; s.lnL = lnL; s.nb = nb; s.dt_bits = dt_bits; s.dt_cap = dt_cap;
    s.stats = stats;
    s.taus = taus; s.taus_base = taus_base;
    s.n_seg = n_seg;
    return s;
  }
};

// Scratch of the radix sort (sized for a given layout).
struct SortWork {
  uint64_t* keys_alt = nullptr;
  uint32_t* vals_alt = nullptr;
  unsigned long long* desc = nullptr;   // [passes][n_tiles][256] look-back words
  uint32_t* hist = nullptr;             // [n_seg][passes][256]
  uint32_t* tickets = nullptr;          // [passes]
  uint32_t* done = nullptr;             // [n_seg] upsweep blocks finished
  size_t zero_head = 0;                 // bytes before desc (zeroed with it per sort)
  void* zero_base = nullptr;
  int max_passes = 0;
  // shape of the digit passes: keys per thread (8 or 16) and multisplit
  // (0: __match_any_sync, 1: ballots); tiles of 256 * ipt keys
  int ipt = 16;
  int rank = 0;
  int64_t n_stiles = 0;
  int64_t* stile_off = nullptr;         // n_seg + 1 tile offsets of that shape
  void* block = nullptr;
};

// choose the pass shape (host offsets are copied; not during stream capture)
cudaError_t sort_set_shape(const SegLayout& L, SortWork& W, int ipt, int rank,
                           cudaStream_t st);

// allocation helpers (stream-ordered); return cudaError_t
cudaError_t alloc_layout(SegLayout& L, const std::vector<int64_t>& sizes,
                         const std::vector<uint64_t>& seeds, const std::vector<double>& lnL,
                         int bin_size, cudaStream_t st);
void free_layout(SegLayout& L, cudaStream_t st);
// keys, zeroed: memory for its keys and counters (n keys and sort_zeroed_bytes;
// the caller's), null: its own
cudaError_t alloc_sort(SortWork& W, const SegLayout& L, int max_passes, cudaStream_t st,
                       uint64_t* keys = nullptr, void* zeroed = nullptr);
size_t sort_zeroed_bytes(const SegLayout& L, int max_passes);
void free_sort(SortWork& W, cudaStream_t st);

// ------------------------------------------------------------- launchers
// Stable LSD radix sort of (keys, vals) within each segment over the 8-bit
// digits [first_pass, first_pass + passes).  When vals_identity is set the
// input values are taken to be the global positions.  After an even number
// of passes the result is in (keys, vals); after an odd number it is in the
// alternate buffers, which *keys_res / *vals_res then name when both are
// given (else it is copied back into keys, vals).
cudaError_t sort_segments(const SegLayout& L, SortWork& W, uint64_t* keys, uint32_t* vals,
                          int first_pass, int passes, bool vals_identity, uint32_t* err,
                          cudaStream_t st, uint64_t** keys_res = nullptr,
                          uint32_t** vals_res = nullptr);

// Order every run of finite keys equal in their bits from `shift` up by
// (key, id of the element: ids_by_val[vals[p] * id_stride]), so that after
// a sort on those bits the (r, id) order holds (shift 0: runs of equal
// radii, ordered by id).
void launch_tiefix(const SegLayout& L, uint64_t* keys, uint32_t* vals,
                   const uint32_t* ids_by_val, int id_stride, uint32_t* err,
                   cudaStream_t st, int shift = 0);

void launch_philox(int64_t n, const uint32_t* ctr, uint64_t seed, uint32_t* out,
                   cudaStream_t st);

// One star between the orbit step and the sorted state, in two records of
// one 32-byte sector each.  RecA goes with the gather after the sort: the new
// radius, its reciprocal, the mass, the id and the star's sort bin.  RecB
// waits for the new potential: the new velocities and c (for a bound star
// Phi_old(r_old) - Phi_old(r_new); for a star escaping in this step its
// energy in the field of the others, Phi_k + m_k / r_k + v^2 / 2), and w,
// Phi_new(r_old), filled in once the new potential is there.
struct alignas(32) RecA {
  double r, x, m;
  uint32_t id, bin;
};
struct alignas(32) RecB {
  double vr, vt, c, w;
};
// (each moves as one 32-byte access: two of 16 bytes fetched a random record's
// sector twice, gather 0.37 -> 0.70 ms with three blocks to an SM)
__device__ __forceinline__ RecA load_rec(const RecA* p) {
  const double4_32a v = *reinterpret_cast<const double4_32a*>(p);
  const unsigned long long u = ubits(v.w);
  RecA a;
  a.r = v.x; a.x = v.y; a.m = v.z; a.id = (uint32_t)u; a.bin = (uint32_t)(u >> 32);
  return a;
}
__device__ __forceinline__ RecB load_rec(const RecB* p) {
  const double4_32a v = *reinterpret_cast<const double4_32a*>(p);
  RecB b;
  b.vr = v.x; b.vt = v.y; b.c = v.z; b.w = v.w;
  return b;
}
__device__ __forceinline__ void store_rec(RecA* p, const RecA& a) {
  *reinterpret_cast<double4_32a*>(p) = make_double4_32a(
      a.r, a.x, a.m,
      __longlong_as_double((long long)(((unsigned long long)a.bin << 32) | a.id)));
}
__device__ __forceinline__ void store_rec(RecB* p, const RecB& b) {
  *reinterpret_cast<double4_32a*>(p) = make_double4_32a(b.vr, b.vt, b.c, b.w);
}

// The counting sort of a timestep.  A star's bin is the shell of the old
// table that its new radius lies in (the orbit step has just found it):
// bins order like radii, and since the distribution of the radii changes
// little in a step a bin holds about one star.  So counting the bins,
// scanning the counts and scattering the stars' indices sorts them up to the
// order inside a bin, which the gather settles by (r, id).  Bins of segment
// c: cbase[c] + s + 1 for the stars in shell s = -1 .. nb - 1, then the
// escapers by id >> esh[c].  Runs of more than kRunMax stars in one bin are
// listed and sorted by a kernel of their own (k_long_runs).
struct BinWork {
  int64_t* cbase = nullptr;             // n_seg + 1 first bins
  int* esh = nullptr;                   // per segment: ids per escaper bin (a shift)
  uint32_t* cnt = nullptr;              // counts, then positions; zero between steps
  unsigned long long* desc = nullptr;   // look-back words of the scan; zero between steps
  uint32_t* ctl = nullptr;              // kCtl words; zero between steps
  uint2* runs = nullptr;                // listed runs of up to kRunTile: first position, length
  uint4* big = nullptr;                 // longer ones: first position, length, their tiles
  std::vector<int64_t> h_cbase;
  int64_t n_bins = 0, n_tiles = 0;      // bins padded to whole scan tiles
};
constexpr int kRunMax = 32;
constexpr int kRunTile = 2048;          // stars of a long run per block
enum : int {
  kCtlScan,   // the scan's tickets
  kCtlRuns,   // listed runs of up to kRunTile
  kCtlBig,    // longer ones
  kCtlTiles,  // their tiles
  kCtlMost,   // tiles of the longest
  kCtlNext,   // k_long_runs' tickets
  kCtlDone,   // tiles it has done, over all passes
  kCtlLeft,   // blocks that have left it
  kCtlWords
};
constexpr int kBinTile = 4096;          // bins per block of the scan
cudaError_t alloc_bins(BinWork& B, const SegLayout& L, cudaStream_t st);
void free_bins(BinWork& B, cudaStream_t st);
// the escapers' bins for the largest id of each segment
cudaError_t set_bin_ids(BinWork& B, const SegLayout& L, const unsigned int* max_id,
                        cudaStream_t st);
// order (n indices): the stars' indices in bin order, the order inside a bin
// left to the gather except in the listed runs, which are in (r, id) order.
// bin (n): each star's bin; counted: the orbit step has counted the bins.
// scratch: n indices; keys, keys_scratch: n keys each (long runs).
void launch_bin_sort(const SegLayout& L, BinWork& B, const uint32_t* bin, const RecA* rec,
                     uint32_t* order, uint32_t* scratch, uint64_t* keys, uint64_t* keys_scratch,
                     bool counted, uint32_t* err, cudaStream_t st);

// keys of the current state (radius_key of r, id)
void launch_make_keys(const SegLayout& L, const double* r, const uint32_t* id, uint64_t* keys,
                      cudaStream_t st);
// records of the current state (for the initial ordering)
void launch_make_records(const SegLayout& L, const double* r, const double* vr,
                         const double* vt, const double* m, const uint32_t* id, RecA* ra,
                         RecB* rb, cudaStream_t st);

// keys = id (for the (r, id) order at initialisation), and radius keys of
// the stars in the order of a permutation
void launch_id_keys(const SegLayout& L, const uint32_t* id, uint64_t* keys, cudaStream_t st);
void launch_rekey_radius(const SegLayout& L, const uint32_t* perm, const double* r,
                         const uint32_t* id, uint64_t* keys, cudaStream_t st);

// records in the order of a permutation -> SoA state (initial ordering)
void launch_gather(const SegLayout& L, const uint32_t* perm, const RecA* ra, const RecB* rb,
                   double* r, double* x, double* vr, double* vt, double* m, uint32_t* id,
                   cudaStream_t st);
// The timestep's gather: r, x, m, id in (r, id) order with the potential's
// per-tile sums over the bound stars (launch_potential with sums_ready then
// skips them); order_out: the star's old index at each new position; r_out and
// x_out must not be r_in (the old radii, still wanted for the energy
// correction).  exact: order_in is in (r, id) order already; else bin order.
// For the escaped stars also r_old (the old radius, +inf for those that
// escaped before) and c.  Rp -> Rout, Ap -> Aout: attributes that go along.
// With bins, their counts and scan words are zeroed for the next step.
void launch_gather_step(const SegLayout& L, BinWork* B, const uint32_t* order_in,
                        const RecA* ra, const RecB* rb, const double* r_in, double* r_out,
                        double* x_out, double* m, uint32_t* id, uint32_t* order_out,
                        double* r_old, double* c, double* tile_m, double* tile_mx,
                        const double* Rp, double* Rout, const double* Ap, double* Aout,
                        bool exact, cudaStream_t st);
struct GridBuild;
// Phi_new(r_old) of every star of the old order into its RecB (w), r_in and
// x_in the old radii and reciprocals (sorted), r, x, phi, node the new table.
// div_form: Eq. 6's division form (FP64 modes; node may be null), else the
// shell slope of the node records.  grid: the grid's values are built beside it.
void launch_phi_old(const SegLayout& L, const double* r_in, const double* x_in, const double* r,
                    const double* x, const double* phi, const double4_32a* node, RecB* rb,
                    bool div_form, cudaStream_t st,
                    const GridBuild* grid = nullptr);
// the largest number of stars whose velocities' kernel ends the step too (see
// launch_velocities)
constexpr int64_t kEndWithVelocities = 1 << 20;
// the new velocities into place, corrected for the changing potential
// (correct false: as they are); then the step is committed: nb, escaper
// statistics and budget (from the gathered r_old and c of the escaped range), dt,
// the per-step counters
void launch_velocities(const SegLayout& L, const uint32_t* order, const RecB* rb,
                       const double* phi, const double* m, double* vr, double* vt, bool correct,
                       const double* r_old,
                       const double* c, uint32_t* step, cudaStream_t st);

// potential: per-tile sums then the tile-local scans (Eqs. 1-5 in scan
// form).  nb_sub: subtract esc_step from nb (after the orbit step).
// With recip (= x), x = 1/r is computed too, with the tiles' sums.
// over_m: phi or Mout shares memory with m, place for place.
// Optional output: Mout (M_k); with tables instead the record {1/r, Phi, r,
// slope} of every star (node: one 32-byte sector per node for the kernels that
// read a few nodes at random; the slope of Eq. 6 across the shell is the FP64
// orbit step's parameter) and the orbit step's index tables.
// The orbit step's index tables as the potential kernel writes them beside
// Phi: the bucket starts and the grid's key shells (their per-segment
// parameters computed before it, from 1/r).
struct TableOut {
  int* start = nullptr;
  const int64_t* boff = nullptr;
  uint32_t* base = nullptr;  // per segment (also read by the orbit step's kernels)
  int4* prm = nullptr;
  int* gshell = nullptr;
  const int64_t* goff = nullptr;
  int4* gprm = nullptr;
  float4* gaux = nullptr;
};
void launch_potential(const SegLayout& L, const double* r, const double* x, const double* m,
                      double* tile_m, double* tile_mx, double* phi, double* Mout, bool nb_sub,
                      cudaStream_t st, bool sums_ready = false, double4_32a* node = nullptr,
                      const TableOut* tables = nullptr, double* recip = nullptr,
                      bool over_m = false);
// node records from the arrays (stage calls)
void launch_make_nodes(int64_t n, const double* r, const double* x, const double* phi,
                       const double* M, double4_32a* node, cudaStream_t st);

void launch_correction(const SegLayout& L, const double* r, const double* x,
                       const double* phi, double* vr, double* vt, const double* r_old,
                       const double* c, bool nb_sub, uint32_t* err, cudaStream_t st,
                       const double* m = nullptr);

// Eq. 7's timesteps of the bins into the segments' timesteps, and the bins'
// densities; with R (stellar radii) or A (semi-major axes) also Eq. 8's
// collision step and Eqs. 9-10's binary steps over the innermost 300 bound stars
void launch_bins(const SegLayout& L, const double* r, const double* vr, const double* vt,
                 const double* m, double* nbin, double pref, cudaStream_t st,
                 const double* R = nullptr, const double* A = nullptr, double x_bb = 0.0,
                 double x_bs = 0.0);

// relaxation of the neighbour pairs; with stellar radii R (may be null)
// pairs may merge (sticky spheres; r and phi: the current table)
void launch_relax(const SegLayout& L, double* vr, double* vt, double* m, const uint32_t* id,
                  const double* nbin, const uint32_t* step, cudaStream_t st, int variant = 0,
                  double* R = nullptr, const double* r = nullptr, const double* phi = nullptr);

struct OrbitStageOut {   // optional per-star outputs of the orbit stage
  double* phi_new = nullptr;
  double* rmin = nullptr;
  double* rmax = nullptr;
  double* F = nullptr;
  int32_t* code = nullptr;
  int32_t* trials = nullptr;
};

// Radius-bucket index of the float table of every segment (mixed mode):
// start[off[c] + b] = first node of segment c whose bucket is >= b.
//
// With it, a potential grid per segment: Phi (float) at the float keys
// key0 + g 2^sh of 1/r, sh = 23 - p for 2^p cells per binade, so that no
// cell straddles a power of two and Phi, linear in 1/r between stars, is
// close to linear in the key inside a cell.
struct BucketArgs {
  const int* start = nullptr;
  const int64_t* off = nullptr;
  const uint32_t* base = nullptr;
  const int4* prm = nullptr;  // shift, bucket count, first and last indexed node
  const float* gphi = nullptr;
  const int64_t* goff = nullptr;
  const int4* gprm = nullptr;    // key0, sh, cells, key of 1/r_0 (as int)
  const float4* gaux = nullptr;  // Phi_0, bound mass, 1/r at key0, interpolation bound
  const double4_32a* node = nullptr; // {1/r, Phi, r, M} per star (potential kernel)
};

struct BucketWork {
  int* start = nullptr;
  int64_t* off = nullptr;
  uint32_t* base = nullptr;
  int4* prm = nullptr;
  float* gphi = nullptr;
  int* gshell = nullptr;  // shell of every grid key (scratch of the grid build)
  int64_t* goff = nullptr;
  int4* gprm = nullptr;
  float4* gaux = nullptr;
  int64_t gcells = 0;  // grid cells over all segments
  double4_32a* node = nullptr;
  void* block = nullptr;
  BucketArgs args() const {
    BucketArgs a;
    a.start = start; a.off = off; a.base = base; a.prm = prm;
    a.gphi = gphi; a.goff = goff; a.gprm = gprm; a.gaux = gaux;
    a.node = node;
    return a;
  }
};

cudaError_t alloc_buckets(BucketWork& B, const SegLayout& L, cudaStream_t st);
void free_buckets(BucketWork& B, cudaStream_t st);
// build the index from t32 over the bound stars (nb - esc_step when nb_sub)
void launch_buckets(const SegLayout& L, const float2* t32, bool nb_sub, BucketWork& B,
                    cudaStream_t st);
// build the potential grid from the FP64 table (x, Phi, the node records)
void launch_grid(const SegLayout& L, const double* x, const double* phi, bool nb_sub,
                 BucketWork& B, cudaStream_t st);
// the grid's values and the seams' slopes (grid_build.cuh)
struct GridBuild {
  const double *x = nullptr, *phi = nullptr;
  BucketArgs B;
  const int* gshell = nullptr;
  float* gphi = nullptr;
  float4* gaux = nullptr;
  double4_32a* node = nullptr;
  int64_t total = 0, n_tiles = 0;  // cells, tiles with a seam to fill
  bool sub = false, fused = false;
};

// The potential with the orbit step's tables in two kernels: the potential
// writing Phi, the node records, bucket starts and grid key shells with the
// segments' parameters, then the grid's values with the slopes at the tile
// seams (with `later` left to launch_phi_old).  The same tables as
// launch_potential + launch_make_nodes + launch_buckets + launch_grid.
void launch_potential_tables(const SegLayout& L, const double* r, const double* x,
                             const double* m, double* tile_m, double* tile_mx, double* phi,
                             bool nb_sub, bool sums_ready, BucketWork& B, cudaStream_t st,
                             GridBuild* later = nullptr, double* recip = nullptr);

// Lanes to a star in the kernels that share a star's samples and trials among
// lanes while there are few stars (k_env_screen, k_sample32: times there).
inline int star_lanes(const SegLayout& L) { return L.n <= 16384 ? 8 : L.n <= 49152 ? 4 : 1; }
// ... in the sampler: one where draws come in sequence.  With more than one, and
// in stream mode, it has one shape, whatever variant is asked for.
inline int sampler_lanes(const SegLayout& L) { return L.taus ? 1 : star_lanes(L); }
inline bool sampler_has_variants(const SegLayout& L) { return !L.taus && sampler_lanes(L) == 1; }
// two lanes to a pair in the relaxation while there are few pairs (k_relax), in one
// shape
inline bool relax_two_lanes(const SegLayout& L) { return !L.taus && L.n_pairs <= 16384; }

// launch_orbit writes the stars' records, and with bins their sort bins (count:
// counted too) or else their sort keys.  precision 1 (mixed): it runs four kernels (turning points,
// FP32 sampler, FP64 continuation of the pending stars, finishing) and
// needs n records orb (E, J, c0 = (r_max + r_min) / 2, c1 = (r_max -
// r_min) / 4, from the turning-point kernel, for the sampling kernels), a
// list of n uint32 (the pending stars) and one uint32 counter, zero before
// and after (as EnvWork's); tp_min,
// tp_max (n doubles each: the turning points) only with the stage outputs
// of dbg (rmin, rmax).
// precision 0 (FP64): the same kernels with FP64 mode's envelope (two more
// kernels, into an EnvWork) and FP64 mode's points, every decision the FP64
// one.  precision 2 (FP64 by bisection): one kernel on the FP64 table.
void launch_slopes(int64_t n, const double* x, const double* phi, double* Menc,
                   cudaStream_t st);
// one diagnostics record per segment (after the step end; K, W in out3)
void launch_diag_ring(const SegLayout& L, const double* out3, const uint32_t* step,
                      const uint32_t* err, double* ring, int cap, cudaStream_t st);
// FP64 mode's envelope F = 1.2 max_j g(s_j): gmax (n doubles) the maximum
// per star; star (n records) the values its evaluations share; the (star,
// sample) pairs that FP32 bounds cannot rule out, each
// evaluated in FP64 by one thread (list: cap entries p << 5 | j); the stars
// whose pairs found the list full (spill: n entries p << 21 | sample mask);
// cnt[0] pairs, cnt[1] spilled stars
struct EnvWork {
  double* gmax = nullptr;
  double4_32a* star = nullptr;  // E, J, c0, c1 of each star with pairs
  uint64_t* list = nullptr;
  uint64_t* spill = nullptr;
  unsigned long long* cnt = nullptr;
  int64_t cap = 0;
  void* block = nullptr;
};
cudaError_t alloc_env(EnvWork& W, int64_t n, cudaStream_t st);
void free_env(EnvWork& W, cudaStream_t st);

void launch_orbit(const SegLayout& L, int precision, int max_trials, const double* r,
                  const double* x, const double* phi, const double* vr,
                  const double* vt, const double* m, const uint32_t* id, const uint32_t* step,
                  uint64_t* keys, RecA* ra, RecB* rb, const OrbitStageOut* dbg, int block,
                  int variant, const BucketArgs& ba, double* tp_min, double* tp_max,
                  uint32_t* plist, uint32_t* pcount, cudaStream_t st,
                  bool with_turning = true, const double* Rv = nullptr, double* Rp = nullptr,
                  const EnvWork* env = nullptr, const double* Av = nullptr,
                  double* Ap = nullptr, double4_32a* orb = nullptr,
                  const BinWork* bins = nullptr, uint32_t* bin = nullptr, bool count = false);
// the turning-point kernel alone (mixed mode; launch_orbit(..., false)
// then runs the sampling kernel only)
void launch_turning(const SegLayout& L, const double* r, const double* x, const double* phi,
                    const double* vr, const double* vt,
                    const BucketArgs& ba, double* tp_min, double* tp_max, double4_32a* orb,
                    int block, cudaStream_t st);
// mixed-mode orbit variants: register caps for 1 (none), 2, 3, 4, 5, 6 and
// 8 resident 256-thread blocks per SM (128, 80, 64, 48, 40 and 32
// registers; the kernel is latency-bound, and occupancy buys more than the
// spills cost)
constexpr int kOrbitVariants = 7;
constexpr int kRelaxVariants = 3;  // relaxation kernel register caps (launch_relax)

// energy diagnostics: per-segment K, W_pair
void launch_energy(const SegLayout& L, const double* r, const double* vr, const double* vt,
                   const double* m, double* tile_m, double* tile_k, double* tile_w,
                   double* out3, cudaStream_t st);
int energy_kernels(const SegLayout& L);  // that it launches
// the mass up to and including every bound star
void launch_masses(const SegLayout& L, const double* m, double* tile_m, double* Mout,
                   cudaStream_t st);

// core diagnostics (Eq. 19) per cluster: out3 = {rho_c, r_c, estimates};
// tiles4: 4 * n_tiles doubles of scratch
void launch_core(const SegLayout& L, const double* r, const double* m, double* tiles4,
                 double* out3, cudaStream_t st);
void launch_lagrange(const SegLayout& L, const double* r, const double* M,
                     const double* fracs, int nf, double* out, cudaStream_t st);

void launch_validate(const SegLayout& L, const double* r, const double* vr,
                     const double* vt, const double* m, bool allow_inf, uint32_t* err,
                     cudaStream_t st);

// nb of every segment = position of its first escaper key (sorted keys)
void launch_nb_from_keys(const SegLayout& L, const uint64_t* keys, cudaStream_t st);
void launch_recip(int64_t n, const double* r, double* x, cudaStream_t st);
void launch_make_t32(int64_t n, const double* x, const double* phi, float2* t32,
                     cudaStream_t st);
void launch_unpack_orbit(int64_t n, const RecA* ra, const RecB* rb, double* r_new,
                         double* vr_new, double* vt_new, cudaStream_t st);
void sort_prepare();
// look-back polls and tie-fix moves before the sort's waits give up (<= 0:
// the defaults), on the current device
cudaError_t set_wait_limits(int spin_polls, long long tie_moves);
void diag_prepare();
void potential_prepare();  // shared-memory limit of the potential kernel

// (r, id) order of staged stars (flag bit 0 set when not) and the largest id
// per segment (maxid: n_seg values, zeroed by the caller)
void launch_order_check(const SegLayout& L, const double* r, const uint32_t* id, uint32_t* flag,
                        unsigned int* maxid, cudaStream_t st);

// stars in (r, id) order: every id of a segment once (a bitmap, zero before;
// bitoff: the segments' first bits), N_bound of the segments
void launch_place(const SegLayout& L, const double* r, const uint32_t* id,
                  const unsigned long long* bitoff, unsigned long long* bitmap, uint32_t* err,
                  cudaStream_t st);
// starting states of the Tausworthe streams (dynamics.cu): slots of
// segment c from base[c] (n_seg + 1 offsets), words: the segment's seeded
// words, P: [4][32][32] jump matrices T^(2^(80 + b))
void launch_taus_init(int64_t slots, int n_seg, const int64_t* base, const uint4* words,
                      const uint32_t* P, uint4* table, cudaStream_t st);
// flag = 1 if a value is negative, infinite or NaN
void launch_check_attr(int64_t n, const double* a, uint32_t* flag, cudaStream_t st);
void launch_check_ids(const SegLayout& L, const uint64_t* sorted_ids, uint32_t* err,
                      cudaStream_t st);

// The first failed index check of each translation unit of a debug build
// since the last call (0: none), cleared; 0 in a release build.
uint32_t debug_site_tu1();
uint32_t debug_site_tu2();
uint32_t debug_site_tu3();
uint32_t debug_site_tu4();
uint32_t debug_site_tu5();
#define CMC_CAT2(a, b) a##b
#define CMC_CAT(a, b) CMC_CAT2(a, b)
#ifdef CMC_DEBUG
#define CMC_DEBUG_SITE_ACCESSOR                                              \
  uint32_t CMC_CAT(debug_site_tu, CMC_TU)() {                                \
    unsigned int v = 0u, z = 0u;                                             \
    cudaMemcpyFromSymbol(&v, g_debug_site, sizeof(v));                       \
    cudaMemcpyToSymbol(g_debug_site, &z, sizeof(z));                         \
    return v;                                                                \
  }
#else
#define CMC_DEBUG_SITE_ACCESSOR \
  uint32_t CMC_CAT(debug_site_tu, CMC_TU)() { return 0u; }
#endif

}  // namespace cmc
