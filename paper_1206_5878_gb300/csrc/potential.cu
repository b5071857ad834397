// Shell potential (section 2.1 step 1, Eqs. 1-5), the energy correction of
// section 2.1 step 6, the diagnostics, and the data movement around the
// sort (payload gather).
//
// The potential is Eq. 1 in scan form, Phi_k = -G (M_k / r_k + S_k) with
// M_k = sum_{i<=k} m_i and S_k = sum_{i>k} m_i / r_i, over the bound stars
// of each segment.  The scan is reduce-then-scan on fixed tiles: one kernel
// writes per-tile sums, the next combines, per tile, the sums of the tiles
// before it (for M) and after it (for S) in a fixed order and scans inside
// the tile.  Every sum is therefore evaluated in the same order on every
// run, so a cluster gives the same bits whether it is advanced alone or in
// an ensemble, and a resumed run repeats an uninterrupted one exactly.
#include <cmath>
#include <cstring>

#include "grid_build.cuh"

namespace cmc {

namespace {

constexpr int kThreads = 256;
constexpr int kPer = kTile / kThreads;  // 16 consecutive elements per thread

__device__ __forceinline__ int64_t nb_eff(const int64_t* nb, const int64_t* esc, int c,
                                          bool sub) {
  int64_t v = nb[c];
  if (sub) v -= esc[c];
  return v;
}

// fixed-shape block reduction of one double per thread (256 threads)
__device__ __forceinline__ double block_sum(double v, double* s) {
  s[threadIdx.x] = v;
  __syncthreads();
  for (int w = kThreads / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) s[threadIdx.x] = s[threadIdx.x] + s[threadIdx.x + w];
    __syncthreads();
  }
  double r = s[0];
  __syncthreads();
  return r;
}

struct TR {
  int seg;
  int64_t lt, nt, seg_begin, begin, end, bound_end;
};

__device__ __forceinline__ TR tile_of(const Seg& S, const int64_t* esc, int64_t t, bool sub) {
  TR R;
  R.seg = seg_find(S.tile_off, S.n_seg, t);
  int64_t t0 = S.tile_off[R.seg];
  R.lt = t - t0;
  R.nt = S.tile_off[R.seg + 1] - t0;
  R.seg_begin = S.off[R.seg];
  int64_t se = S.off[R.seg + 1];
  R.begin = R.seg_begin + R.lt * kTile;
  R.end = R.begin + kTile < se ? R.begin + kTile : se;
  R.bound_end = R.seg_begin + nb_eff(S.nb, esc, R.seg, sub);
  return R;
}

// --------------------------------------------------------------- gather
__global__ void k_make_keys(int64_t n, const double* r, const uint32_t* id, uint64_t* keys) {
  pdl_enter();
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p < n) keys[p] = radius_key(r[p], id[p]);
}

__global__ void k_make_records(int64_t n, const double* r, const double* vr, const double* vt,
                               const double* m, const uint32_t* id, RecA* ra, RecB* rb) {
  pdl_enter();
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const double rr = r[p];
  RecA A;
  A.r = rr; A.x = lt_inf(rr) ? div_rn(1.0, rr) : 0.0; A.m = m[p]; A.id = id[p]; A.bin = 0u;
  store_rec(ra + p, A);
  RecB B;
  B.vr = vr[p]; B.vt = vt[p]; B.c = 0.0; B.w = 0.0;
  store_rec(rb + p, B);
}

__global__ void k_id_keys(int64_t n, const uint32_t* id, uint64_t* keys) {
  pdl_enter();
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p < n) keys[p] = (uint64_t)id[p];
}

__global__ void k_rekey_radius(int64_t n, const uint32_t* perm, const double* r,
                               const uint32_t* id, uint64_t* keys) {
  pdl_enter();
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  uint32_t q = perm[p];
  // (out of range only after a reported sort failure)
  keys[p] = (int64_t)q < n ? radius_key(r[q], id[q]) : ~0ull;
}

__global__ void k_gather(int64_t n, const uint32_t* perm, const RecA* ra, const RecB* rb,
                         double* r, double* x, double* vr, double* vt, double* m,
                         uint32_t* id) {
  pdl_enter();
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const uint32_t v = perm[p];
  if ((int64_t)v >= n) return;  // only after a reported sort failure
  const RecA A = load_rec(ra + v);
  const RecB B = load_rec(rb + v);
  r[p] = A.r; x[p] = A.x; vr[p] = B.vr; vt[p] = B.vt; m[p] = A.m; id[p] = A.id;
}

// The timestep's gather, a block per tile of kTile new positions or (kSpan <
// kTile) per part of one.  Each star
// counts the members of its bin's run that come before it in (r, id) order --
// runs hold one or two stars, so a few neighbours -- and writes its record to
// its place.  A star belongs to the block its place falls in, so the block walks
// its span and kRunMax positions on each side: a run of up to kRunMax stars
// across its edge is seen whole.  Longer runs are in order already
// (k_long_runs).
//
// Bound by the random 32-byte reads of the records (0.215 ms at N = 1e7 for
// those and the writes alone).  The walk is a pipeline of sub-tiles of one star
// per thread: while the star of sub-tile k - 1 looks at its neighbours (radii
// and bins of sub-tiles k - 2 .. k in a shared-memory ring of four), the record
// of k + 1 and the index of k + 2 are on their way, so that the reads go on
// through the ranking: 0.31 ms (0.42 with the whole tile loaded first).
//
// The potential's per-tile sums of m and m x (k_tile_sums over the bound stars
// after the orbit step) come from the values just written, in the same
// striped element order and tree, so they are the same sums: half the block
// sums m, the other half m x.  Of a tile in parts, the block that finishes last
// (a counter per tile) takes them.
// Blocks of 512 threads, three to an SM (40 registers: a spill would miss the
// L1 under the random reads, which made the kernel twice as slow); while there
// are fewer tiles than SMs blocks of 1024, whose walk is half as long; with few
// tiles a tile in eight parts whose walk is one sub-tile (the stage at 10^4, 10^5,
// 2 x 10^5, 3 x 10^5, 6 x 10^5 stars 19.1, 20.4, 25.8, 31.4, 46.4 us against 30.9,
// 32.1, 32.6, 32.6, 33.0; in sixteen parts 18.6, 24.4, 30.6, 37.6, 61.4).
constexpr int64_t kGatFewTiles = 152, kGatPartTiles = 64;
constexpr int kGatSpan = 512;

struct GatherOut {
  double *r, *x, *m;
  uint32_t *id, *order;
  double *r_old, *c;        // escaped stars only
  double *tile_m, *tile_mx;
  const double *Rp, *Ap;    // attributes that go along (may be null)
  double *R, *A;
};

template <bool kExact, int kSpan, int kGatThreads>
__global__ void __launch_bounds__(kGatThreads, kGatThreads == 512 ? 3 : kGatThreads == 1024 ? 1 : 2)
    k_gather_step(
    Seg S, const int64_t* esc, int64_t n, const uint32_t* order, const RecA* ra, const RecB* rb,
    const double* r_in, GatherOut O, uint32_t* cnt, int64_t n_bins, unsigned long long* desc,
    int64_t n_desc, uint32_t* ctl, uint32_t* done) {
  pdl_enter();
  constexpr int kParts = kTile / kSpan;
  constexpr int kGatWin = kSpan + 2 * kRunMax;
  constexpr int kGatSub = (kGatWin + kGatThreads - 1) / kGatThreads;  // the last one partial
  constexpr int kGatRing = kParts > 1 ? 2048 : 4 * kGatThreads;
  static_assert(kParts == 1 || (kGatSub + 1) * kGatThreads <= kGatRing, "the ring does not wrap");
  static_assert(kRunMax < kGatThreads, "a run's reach is the next sub-tile");
  static_assert(kGatThreads >= 2 * kThreads && kGatThreads <= 1024, "two trees of kThreads");
  __shared__ unsigned long long s_r[kGatRing];
  __shared__ uint32_t s_bin[kGatRing];
  __shared__ double s_red[2 * kThreads];
  const int t = threadIdx.x;
  const int64_t tile = blockIdx.x / kParts;
  TR R = tile_of(S, esc, tile, true);
  const int tlen = (int)(R.end - R.begin);
  // this block's part of the tile; window element w = its position w - kRunMax,
  // within the segment
  const int c0 = (int)(blockIdx.x % kParts) * kSpan;
  const int len = tlen - c0 < kSpan ? tlen - c0 : kSpan;  // (<= 0 in a last tile's empty parts)
  const int64_t pb = R.begin + c0;
  const int64_t w0 = pb - kRunMax;
  const int wa = w0 < R.seg_begin ? (int)(R.seg_begin - w0) : 0;
  const int64_t we = S.off[R.seg + 1] - w0;
  const int wb = we < kGatWin ? (int)we : kGatWin;
  constexpr uint32_t kNone = 0xFFFFFFFFu;  // no star (and a bin that no star has)
  auto index_of = [&](int w) {
    uint32_t v = w >= wa && w < wb ? order[w0 + w] : kNone;
    return (int64_t)v < n ? v : kNone;  // (out of range only after a reported sort failure)
  };
  RecA A;
  A.bin = kNone;
  double px = 0.0, pm = 0.0;  // the star being placed (its r and bin are in the ring)
  uint32_t pid = 0u, pv = kNone;
  uint32_t v = index_of(t), v1 = index_of(t + kGatThreads);
  if (v != kNone) A = load_rec(ra + v);
#pragma unroll 1
  for (int k = 0; k <= kGatSub; ++k) {
    const int w = k * kGatThreads + t;
    RecA A1;
    A1.bin = kNone;
    if (v1 != kNone) A1 = load_rec(ra + v1);
    const uint32_t v2 = index_of(w + 2 * kGatThreads);
    s_r[w & (kGatRing - 1)] = ubits(A.r);
    s_bin[w & (kGatRing - 1)] = A.bin;
    if (!kExact) __syncthreads();
    // the star of the sub-tile before: to the start of its run plus the
    // members before it
    if (pv != kNone) {
      const int wp = w - kGatThreads;
      const unsigned long long r = s_r[wp & (kGatRing - 1)];
      int f = wp;
      if (!kExact) {
        const uint32_t b = s_bin[wp & (kGatRing - 1)];
        auto bin_at = [&](int q) { return s_bin[q & (kGatRing - 1)]; };
        auto r_at = [&](int q) { return s_r[q & (kGatRing - 1)]; };
        int before = 0, left = 0, right = 0, equal = 0;
        auto look = [&](int q) {
          const unsigned long long rq = r_at(q);
          const bool eq = rq == r && ra[order[w0 + q]].id < pid;
          before += rq < r || eq;
          equal += eq;
        };
        for (int q = wp - 1; q >= 0 && left < kRunMax && bin_at(q) == b; --q, ++left) look(q);
        for (int q = wp + 1; q < kGatWin && left + right < kRunMax && bin_at(q) == b; ++q, ++right)
          look(q);
        if (left + 1 + right <= kRunMax) f = wp - left + before;
        else equal = left > 0 && r_at(wp - 1) == r ? (left > 1 && r_at(wp - 2) == r ? 2 : 1) : 0;
        // a group of equal finite radii counts once, at its second star
        if (equal == 1 && r < kInfBits && f >= kRunMax && f < kRunMax + len)
          stat_add(S.stats, R.seg, kStTies, 1ull);
      }
      f -= kRunMax;
      if (f >= 0 && f < len) {
        const int64_t p = pb + f;
        O.r[p] = __longlong_as_double((long long)r);
        O.x[p] = px;
        O.m[p] = pm;
        O.id[p] = pid;
        O.order[p] = pv;
        if (O.R) O.R[p] = O.Rp[pv];
        if (O.A) O.A[p] = O.Ap[pv];
        if (p >= R.bound_end) {
          // escaped: for the step's budget, the old radius of those that left
          // in this step, and c
          O.r_old[p] = (int64_t)pv - R.seg_begin < S.nb[R.seg]
                           ? r_in[pv]
                           : __longlong_as_double((long long)kInfBits);
          O.c[p] = rb[pv].c;
        }
      }
    }
    px = A.x;
    pm = A.m;
    pid = A.id;
    pv = v;
    A = A1;
    v = v1;
    v1 = v2;
  }
  // the tile's sums, by its last block
  bool last = true;
  if (kParts > 1) {
    __shared__ bool s_last;
    __threadfence();
    __syncthreads();
    if (t == 0) {
      s_last = atomicAdd(done + tile, 1u) == kParts - 1u;
      if (s_last) done[tile] = 0u;
      __threadfence();
    }
    __syncthreads();
    last = s_last;
  } else {
    __syncthreads();
  }
  if (last) {
    const int h = t & (kThreads - 1);
    const bool sums = t < 2 * kThreads, second = t >= kThreads;
    const int64_t bl = R.bound_end - R.begin;
    const int lb = bl < tlen ? (int)(bl < 0 ? 0 : bl) : tlen;
    const double* tm = O.m + R.begin;
    const double* tx = O.x + R.begin;
    double a = 0.0;
    if (sums) {
#pragma unroll(kParts > 1 ? kPer : 8)
      for (int i = 0; i < kPer; ++i) {
        const int e = i * kThreads + h;
        if (e < lb) {
          if (kParts > 1) {
            // (past the L1: other blocks wrote them; one block at work: the
            // products on the integer pipes)
            const double me = __ldcg(tm + e);
            a = a + (second ? mul_rn(me, __ldcg(tx + e)) : me);
          } else {
            a = a + (second ? tm[e] * tx[e] : tm[e]);
          }
        }
      }
      s_red[t] = a;
    }
    __syncthreads();
    // block_sum's tree, its last levels in a warp's registers
#pragma unroll
    for (int w = kThreads / 2; w >= 32; w >>= 1) {
      if (sums && h < w) {
        a = a + s_red[t + w];
        s_red[t] = a;
      }
      __syncthreads();
    }
    if (sums && h < 32) {
#pragma unroll
      for (int w = 16; w > 0; w >>= 1) a = a + __shfl_down_sync(0xFFFFFFFFu, a, w);
      if (h == 0) (second ? O.tile_mx : O.tile_m)[tile] = a;
    }
  }
  // the bins' counts and the scan's words, zero again for the next step
  if (cnt) {
    const int64_t step = (int64_t)gridDim.x * kGatThreads;
    const int64_t g = (int64_t)blockIdx.x * kGatThreads + t;
    uint4* c4 = reinterpret_cast<uint4*>(cnt);
    for (int64_t i = g; i < n_bins / 4; i += step) c4[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int64_t i = g; i < n_desc; i += step) desc[i] = 0ull;
    if (g < kCtlWords) ctl[g] = 0u;
  }
}

// ------------------------------------------- the energy correction's halves
// Phi_new at the old radii.  The old radii are sorted as the new table is, so
// a stretch of old stars meets one stretch of the new table: its ends are found
// by two warps (32 probes a round), its radii are staged, and each star
// searches them there (a dozen probes of shared memory, four stars a thread
// abreast) and reads one node next to its neighbours'.  Where the stretch is
// too long to stage, the search runs on the table.  With the velocities'
// kernel 0.42 ms at N = 1e7, 18 us at 1e5; the one kernel before them, in the new
// order with a random search through the bucket index per star, 0.44 ms.  With one
// star a thread there are four times the blocks: faster while they find idle
// SMs (both kernels at 10^4, 10^5, 2 x 10^5 stars 12.3, 14.3, 17.7 us against
// 16.4, 18.4, 20.5), slower above (7 x 10^5: 39.3 against 37.5).
// The grid's values (grid_build) go in the first blocks of this kernel: both need
// the potential only, and alone they took 7 us of mostly latency (potential,
// correction and end of 10^3, 10^5, 10^6 stars 38.7, 53.4, 124.3 us with both and the
// step's end in kernels of their own, 33.2, 45.7, 117.5 so).
constexpr int kPoThreads = 256;
constexpr int kPoPer = 4;     // stars per thread, 1 while there are few tiles
constexpr int64_t kPoFewTiles = 76;
constexpr int kPoWin = 2048;  // staged radii at most
static_assert(kTile % (kPoThreads * kPoPer) == 0, "whole chunks in a tile");

// largest i in [0, nb) with r[i] <= q, else -1, by one warp
__device__ __forceinline__ int64_t warp_shell(const double* r, int64_t nb, double q) {
  const long long qb = dbits(q);
  const int lane = threadIdx.x & 31;
  int64_t lo = -1, hi = nb;
  while (hi - lo > 1) {
    const int64_t span = hi - lo;
    const int64_t m = lo + (span * (lane + 1)) / 33;
    const bool below = m <= lo || (m < hi && dbits(r[m]) <= qb);
    const unsigned k = (unsigned)__popc(__ballot_sync(0xffffffffu, below));
    // the first k probes are at or below q (probes rise with the lane)
    const int64_t nlo = k == 0 ? lo : lo + (span * k) / 33;
    const int64_t nhi = k == 32 ? hi : lo + (span * (k + 1)) / 33;
    lo = nlo > lo ? nlo : lo;
    hi = nhi < hi ? nhi : hi;
  }
  return lo;
}

template <bool kDiv, int kPer>
__global__ void __launch_bounds__(kPoThreads) k_phi_old(Seg S, const int64_t* esc,
                                                        const double* r_in, const double* x_in,
                                                        const double* r, const double* x,
                                                        const double* phi,
                                                        const double4_32a* node, RecB* rb,
                                                        GridBuild G, unsigned grid_blocks) {
  pdl_enter();
  if (blockIdx.x < grid_blocks) {
    grid_build(S, esc, G, (int64_t)blockIdx.x * kPoThreads + threadIdx.x);
    return;
  }
  const unsigned chunk = blockIdx.x - grid_blocks;
  __shared__ long long po_r[kPoWin];
  __shared__ int64_t s_lo, s_hi;
  const int t = threadIdx.x;
  constexpr int kPoChunk = kPoThreads * kPer;  // the block's stars
  constexpr int kSub = kTile / kPoChunk;
  TR R = tile_of(S, esc, chunk / kSub, false);
  // the old order's bound stars in this chunk; the new table
  const int64_t begin = R.begin + (int64_t)(chunk % kSub) * kPoChunk;
  int64_t end = begin + kPoChunk < R.end ? begin + kPoChunk : R.end;
  end = end < R.bound_end ? end : R.bound_end;
  if (begin >= end) return;
  const int64_t sb = R.seg_begin, nb = S.nb[R.seg] - esc[R.seg];
  if (nb <= 0) return;
  double ro[kPer], xo[kPer];
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const int64_t p = begin + j * kPoThreads + t;
    ro[j] = p < end ? r_in[p] : 0.0;
    xo[j] = p < end ? x_in[p] : 0.0;
  }
  if (t < 64) {
    const int64_t k = warp_shell(r + sb, nb, r_in[t < 32 ? begin : end - 1]);
    if (t == 0) s_lo = k;
    if (t == 32) s_hi = k;
  }
  __syncthreads();
  const int64_t lo0 = s_lo, hi0 = s_hi + 1;  // shells lo0 .. hi0 - 1
  const int64_t first = lo0 < 0 ? 0 : lo0;
  const int staged = (int)(hi0 - first < kPoWin ? hi0 - first : kPoWin + 1);
  int64_t at[kPer];
  if (staged <= kPoWin) {
    for (int i = t; i < staged; i += kPoThreads) po_r[i] = dbits(r[sb + first + i]);
    __syncthreads();
    int lo[kPer], hi[kPer];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      lo[j] = lo0 < 0 ? -1 : 0;  // (r[lo0] is not above the chunk's first star)
      hi[j] = staged;
    }
    // every star's bracket shrinks alike: staged or staged + 1 candidates
    for (int width = staged + 1; width > 1; width = (width + 1) >> 1) {
#pragma unroll
      for (int j = 0; j < kPer; ++j) {
        const int mid = (lo[j] + hi[j]) >> 1;
        if (mid > lo[j]) {
          if (po_r[mid] <= dbits(ro[j])) lo[j] = mid; else hi[j] = mid;
        }
      }
    }
#pragma unroll
    for (int j = 0; j < kPer; ++j) at[j] = first + lo[j];
  } else {
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      int64_t lo = lo0, hi = hi0;
      while (hi - lo > 1) {
        const int64_t mid = lo + ((hi - lo) >> 1);
        if (dbits(r[sb + mid]) <= dbits(ro[j])) lo = mid; else hi = mid;
      }
      at[j] = lo;
    }
  }
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const int64_t p = begin + j * kPoThreads + t;
    if (p >= end) continue;
    const int64_t i = at[j];
    double pn;
    if (!kDiv) {
      const int64_t q = sb + (i < 0 ? 0 : i);
      const double4_32a nd = node[q];
      // (a seam's slope as the grid's blocks compute it, which may not have yet)
      const double w = i >= 0 && i % kTile == kTile - 1 && i + 1 < nb
                           ? div_rn(phi[q + 1] - nd.y, nd.x - x[q + 1])
                           : nd.w;
      pn = i < 0 ? nd.y : nd.y + w * (nd.x - xo[j]);
    } else {
      const int64_t q = sb + (i < 0 ? 0 : i);
      const double pj = phi[q];
      pn = pj;
      if (i >= 0) {
        const double xj = x[q];
        double xj1 = 0.0, pj1 = 0.0;
        if (i + 1 < nb) {
          xj1 = x[q + 1];
          pj1 = phi[q + 1];
        }
        const double den = xj - xj1;
        if (pos_num(den)) pn = pj + div_rn(xj - xo[j], den) * (pj1 - pj);
      }
    }
    rb[p].w = pn;
  }
}

// The new velocities into the new order: T' = T + 1/2 [(Phi_new(r_old) -
// Phi_new(r_new)) - (Phi_old(r_old) - Phi_old(r_new))], clamped at 0; both
// components scaled by sqrt(T'/T) (section 2.1 step 6).
// The kernel also ends the step: its first n_seg blocks sum what the stars that
// escaped in this step take with them (the escaped range's entries with a finite
// r_old; earlier escapers carry r_old = inf), mass and energy m_k e_k (e_k in c) in
// a fixed order, into the segments' budgets (section 4.2), and its last block to
// finish turns the segments' counters over.  E.done null: not here (a launch
// without stars follows).
struct StepEnd {
  int64_t* esc;
  uint64_t* dt_last;
  uint32_t* step;
  const double *r_old, *e;
  double* esc_me;
  uint32_t* done;  // blocks finished; zero between kernels; null: no end of the step
};

__device__ __forceinline__ void escapers_of(const Seg& S, const StepEnd& E, const double* m, int c) {
  __shared__ double s_m[256], s_e[256];
  const int t = threadIdx.x;
  const int64_t ne = E.esc[c];
  if (ne <= 0) return;
  const int64_t nb_new = S.nb[c] - ne;
  double dm = 0.0, de = 0.0;
  for (int64_t p = S.off[c] + nb_new + t; p < S.off[c + 1]; p += 256)
    if (isfinite(E.r_old[p])) {
      dm += m[p];
      de += m[p] * E.e[p];
    }
  s_m[t] = dm;
  s_e[t] = de;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (t < w) {
      s_m[t] += s_m[t + w];
      s_e[t] += s_e[t + w];
    }
    __syncthreads();
  }
  if (t == 0) {
    E.esc_me[2 * c] += s_m[0];
    E.esc_me[2 * c + 1] += s_e[0];
  }
}

// (32 registers, eight blocks an SM: with 34 and six 206 us at N = 1e7 against 182.)
template <bool kCorrect>
__global__ void __launch_bounds__(256, 8) k_velocities(Seg S, int64_t n, const uint32_t* order,
                                                    const RecB* rb, const double* phi,
                                                    const double* m, double* vr, double* vt,
                                                    StepEnd E) {
  pdl_enter();
  const int64_t p = (int64_t)((int)blockIdx.x - (E.done ? S.n_seg : 0)) * 256 + threadIdx.x;
  if (p < 0) {
    escapers_of(S, E, m, blockIdx.x);
  } else if (p < n) {
    const uint32_t v = order[p];
    if ((int64_t)v < n) {  // (not below only after a reported sort failure)
      const RecB B = load_rec(rb + v);
      double a = B.vr, b = B.vt;
      if (kCorrect) {
        const int c = seg_find(S.off, S.n_seg, p);
        if (p - S.off[c] < S.nb[c] - E.esc[c]) {
          // (two of the four products on the integer pipes: the FP64 pipe bounds
          // this kernel)
          const double Tk = scale_down<1>(mul_rn(a, a) + b * b);
          const double dnew = B.w - phi[p];
          double Tp = Tk + scale_down<1>(dnew - B.c);
          if (lt0(Tp)) {
            clamp_energy_add(S.stats, c, m[p], Tp);
            stat_add(S.stats, c, kStClamps, 1ull);
            Tp = 0.0;
          }
          if (pos_num(Tk)) {
            const double f = sqrt_rn(div_rn(Tp, Tk));
            a = mul_rn(a, f);
            b = b * f;
          }
        }
      }
      vr[p] = a;
      vt[p] = b;
    }
  }
  if (!E.done) return;
  __shared__ bool s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(E.done, 1u) == gridDim.x - 1u;
    if (s_last) *E.done = 0u;
    __threadfence();
  }
  __syncthreads();
  if (!s_last) return;
  for (int c = threadIdx.x; c < S.n_seg; c += 256) {
    const int64_t ne = E.esc[c];
    E.dt_last[c] = S.dt_bits[c];
    S.nb[c] = S.nb[c] - ne;
    // the stars merged away in this step (sticky spheres) left with the
    // escapers; they are counted as collisions, not as escapes
    unsigned long long* st = S.stats + (size_t)c * kStStride;
    const unsigned long long merged = st[kStCollisions] - st[kStCollisionsSeen];
    st[kStCollisionsSeen] = st[kStCollisions];
    st[kStEscaped] += (unsigned long long)ne - merged;
    E.esc[c] = 0;
    S.dt_bits[c] = 0x7FF0000000000000ull;
    if (c == 0) *E.step += 1u;
  }
}

// ------------------------------------------------------------ potential
// per-tile sums of m and m x (striped, coalesced loads; fixed tree).
// kSumsRecip: x = 1/r of every star is computed here too, from r in x's place.
// kSumsMass: of m alone.  The products and quotients are taken by all threads, on
// the integer pipes; the sums run from shared memory, m's by one half of the
// block, m x's by the other.  Two blocks of 64 registers an SM (three spill).
// cmc_potential on 4 x 10^6 stars: reciprocals and sums in two kernels, the sums
// by one thread for both, took 76 us, this kernel half of it.
enum { kSumsOfX, kSumsRecip, kSumsMass };
constexpr int kSumsThreads = 2 * kThreads;
template <int kKind>
__global__ void __launch_bounds__(kSumsThreads, 2) k_tile_sums(Seg S, const int64_t* esc, bool sub,
                                                            const double* x, const double* m,
                                                            double* tile_m, double* tile_mx,
                                                            double* x_out) {
  pdl_enter();
  constexpr bool kBoth = kKind != kSumsMass;
  extern __shared__ double smem[];
  double* s_m = smem;
  double* s_mx = smem + (kBoth ? kTile : 0);
  __shared__ double s_red[kSumsThreads];
  TR R = tile_of(S, esc, blockIdx.x, sub);
  const int t = threadIdx.x, h = t & (kThreads - 1);
  const bool second = t >= kThreads;
  double mv[kTile / kSumsThreads], xv[kTile / kSumsThreads];
#pragma unroll
  for (int j = 0; j < kTile / kSumsThreads; ++j) {
    const int64_t p = R.begin + j * kSumsThreads + t;
    const bool in = p < R.end && p < R.bound_end;
    mv[j] = in ? m[p] : 0.0;
    if (kBoth) xv[j] = (kKind == kSumsRecip ? p < R.end : in) ? x[p] : 1.0;
  }
#pragma unroll
  for (int j = 0; j < kTile / kSumsThreads; ++j) {
    const int e = j * kSumsThreads + t;
    if (kKind == kSumsRecip) {
      xv[j] = div_rn(1.0, xv[j]);
      if (R.begin + e < R.end) x_out[R.begin + e] = xv[j];
    }
    s_m[e] = mv[j];  // (0 where there is no bound star: the sums stay as they are)
    if (kBoth) s_mx[e] = R.begin + e < R.bound_end ? mul_rn(mv[j], xv[j]) : 0.0;
  }
  __syncthreads();
  // half the block sums m, the other half m x: 16 striped elements a thread,
  // then a tree
  double a = 0.0;
  if (kBoth || !second) {
    const double* q = second ? s_mx : s_m;
#pragma unroll 4
    for (int i = 0; i < kPer; ++i) a = a + q[i * kThreads + h];
  }
  s_red[t] = a;
  __syncthreads();
#pragma unroll
  for (int w = kThreads / 2; w >= 32; w >>= 1) {
    if (h < w) {
      a = a + s_red[t + w];
      s_red[t] = a;
    }
    __syncthreads();
  }
  if (h < 32) {
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) a = a + __shfl_down_sync(0xFFFFFFFFu, a, w);
    if (h == 0 && (kBoth || !second)) (second ? tile_mx : tile_m)[blockIdx.x] = a;
  }
}

template <int kKind>
void launch_tile_sums(const SegLayout& L, bool nb_sub, const double* x, const double* m,
                      double* tile_m, double* tile_mx, double* x_out, cudaStream_t st) {
  launch_k(k_tile_sums<kKind>, (unsigned)L.n_tiles, kSumsThreads,
           sizeof(double) * kTile * (kKind == kSumsMass ? 1 : 2), st, L.dev(), L.esc_step, nb_sub,
           x, m, tile_m, tile_mx, x_out);
}

// The potential kernel runs 512 threads on a tile, 8 consecutive elements
// each, so that two tiles' worth of warps (32) share an SM; its shared
// arrays pad one double per 8 (a thread's run of 8 sits 9 words from its
// neighbour's, free of bank conflicts within each half-warp).
// With few tiles the blocks share a tile, up to 16 to one: each takes the tile's
// integer sums by itself (they are exact, so the same in every block) and
// finishes its part of the stars.  Up to two blocks per SM that way: one block
// per tile leaves most SMs idle (the potential stage of 10^4, 10^5 stars 42, 42 us
// against 26, 29; at 245 tiles and more a second block per tile only adds the
// sums' work, 70.2 us against 71.7).  Where the output lies over the masses, one
// block a tile: another block of the tile may not have read them yet.
constexpr int kPotParts = 4;    // log2
constexpr int kPotBlocks = 304;
constexpr int kPotThreads = 512;
constexpr int kPotPer = kTile / kPotThreads;
constexpr int kPotWarps = kPotThreads / 32;
__device__ __forceinline__ int pad8(int e) { return e + (e >> 3); }
constexpr int kPad8N = kTile + kTile / 8;

// fixed-order block sums of two values over kPotThreads threads: a tree in each
// warp, then a tree over the warp totals in the first warp (a, b: kPotWarps + 1
// slots each).  A warp of zeros skips its tree, so a few tiles cost few FP64
// additions (16 cycles each on one SM's pipe).
__device__ __forceinline__ double tree_sum_pot(double v, int o) {
  if (!__any_sync(0xFFFFFFFFu, (ubits(v) << 1) != 0ull)) return 0.0;
  for (; o > 0; o >>= 1) v = v + __shfl_down_sync(0xFFFFFFFFu, v, o);
  return v;
}
__device__ __forceinline__ void block_sums_pot(double& u, double& v, double* a, double* b) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  u = tree_sum_pot(u, 16);
  v = tree_sum_pot(v, 16);
  if (lane == 0) a[w] = u, b[w] = v;
  __syncthreads();
  if (w < 2) {
    double* q = w ? b : a;
    const double z = tree_sum_pot(lane < kPotWarps ? q[lane] : 0.0, kPotWarps / 2);
    if (lane == 0) q[kPotWarps] = z;
  }
  __syncthreads();
  u = a[kPotWarps];
  v = b[kPotWarps];
}

// Fixed point for the sums inside a tile: v >= 0 as round(v 2^S) in 64
// bits, S = 49 - (the largest unbiased exponent among the tile's values),
// so that a sum of 4096 values stays below 2^62; the largest values keep
// 50 significant bits, the sums are then exact (and independent of their
// order), and only the conversion back rounds.  Integer instructions only:
// the FP64 pipe is left to the products.
__device__ __forceinline__ int exp_of(double v) {  // biased exponent (0 for zero)
  return (int)((ubits(v) >> 52) & 0x7FFull);
}

__device__ __forceinline__ long long fix_of(double v, int S) {
  const unsigned long long u = ubits(v);
  const int e = (int)((u >> 52) & 0x7FFull);
  if (e == 0) return 0;  // zero (and subnormals, far below any sum here)
  const unsigned long long mant = (u & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const int sh = e - 1075 + S;  // v = mant 2^(e - 1075); sh <= -3 for the largest
  if (sh < -60) return 0;
  const int d = -sh;
  // round to nearest, ties to even (d in [3, 60]; the rest in the top bits)
  const unsigned long long q = mant >> d, rem = (mant << (64 - d)) | (q & 1ull);
  return (long long)(q + (rem > (1ull << 63) ? 1ull : 0ull));
}

// V 2^-S (V >= 0) as the nearest double, ties to even
__device__ __forceinline__ double dbl_of_fix(long long V, int S) {
  if (V <= 0) return 0.0;
  const unsigned long long a = (unsigned long long)V;
  int top = 63 - __clzll((long long)a);
  unsigned long long m;
  if (top <= 52) {
    m = a << (52 - top);
  } else {
    const int d = top - 52;
    m = a >> d;
    const unsigned long long rem = (a << (64 - d)) | (m & 1ull);
    if (rem > (1ull << 63)) ++m;
    if (m >> 53) {
      m >>= 1;
      ++top;
    }
  }
  return __longlong_as_double(
      (long long)(((unsigned long long)(top - S + 1023) << 52) | (m & 0xFFFFFFFFFFFFFull)));
}

// the largest of one int per thread over kPotThreads threads
__device__ __forceinline__ int block_max_pot(int v, int* w17) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  v = (int)__reduce_max_sync(0xFFFFFFFFu, (unsigned)v);
  if (lane == 0) w17[w] = v;
  __syncthreads();
  int r = 0;
#pragma unroll
  for (int i = 0; i < kPotWarps; ++i) r = w17[i] > r ? w17[i] : r;
  __syncthreads();
  return r;
}

// exclusive forward scan of vm and backward scan of vs (64-bit integers)
// over kPotThreads threads: inclusive scans inside each warp by shuffles,
// the 16 warp totals scanned by one warp, then (totals of the warps before
// or after) + (lanes before or after in the warp)
__device__ __forceinline__ void block_scans_fix(long long vm, long long vs, long long* wm,
                                                long long* ws, long long& pre_m,
                                                long long& suf_s) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  long long a = vm, b = vs;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long ua = __shfl_up_sync(0xFFFFFFFFu, a, o);
    const long long db = __shfl_down_sync(0xFFFFFFFFu, b, o);
    if (lane >= o) a = ua + a;
    if (lane + o < 32) b = b + db;
  }
  const long long ea = __shfl_up_sync(0xFFFFFFFFu, a, 1);
  const long long eb = __shfl_down_sync(0xFFFFFFFFu, b, 1);
  if (lane == 31) wm[w] = a;
  if (lane == 0) ws[w] = b;
  __syncthreads();
  if (w == 0) {
    long long ta = lane < kPotWarps ? wm[lane] : 0ll;
    long long tb = lane < kPotWarps ? ws[lane] : 0ll;
#pragma unroll
    for (int o = 1; o < kPotWarps; o <<= 1) {
      const long long ua = __shfl_up_sync(0xFFFFFFFFu, ta, o);
      const long long db = __shfl_down_sync(0xFFFFFFFFu, tb, o);
      if (lane >= o) ta = ua + ta;
      if (lane + o < kPotWarps) tb = tb + db;
    }
    const long long xa = __shfl_up_sync(0xFFFFFFFFu, ta, 1);
    const long long xb = __shfl_down_sync(0xFFFFFFFFu, tb, 1);
    __syncwarp();
    if (lane < kPotWarps) {
      wm[lane] = lane > 0 ? xa : 0ll;
      ws[lane] = lane + 1 < kPotWarps ? xb : 0ll;
    }
  }
  __syncthreads();
  pre_m = lane > 0 ? wm[w] + ea : wm[w];
  suf_s = lane < 31 ? ws[w] + eb : ws[w];
  __syncthreads();
}

// The index tables' parameters of a segment of nb bound stars (x: its 1/r, from
// the innermost star out).  Buckets: the indexed node range, the smallest shift
// that fits its range of float keys into cap buckets, their count; base = the
// key of the first indexed node.  Grid: the finest 2^p cells per binade (p <= 10)
// that fit cap.
__device__ __forceinline__ int4 bucket_params_of(const double* x, int64_t nb, int64_t cap,
                                                 uint32_t& base) {
  base = 0;
  if (nb <= 0) return make_int4(0, 0, 0, -1);
  const int tail = nb >= 4096 ? (int)(nb >> 10) : 0;
  const int lo = tail, hi = (int)nb - 1 - tail;
  const uint32_t b0 = __float_as_uint(f32_rn(x[lo])), b1 = __float_as_uint(f32_rn(x[hi]));
  const uint32_t span = b0 >= b1 ? b0 - b1 : 0u;
  int bs = 0;
  while ((int64_t)(span >> bs) + 1 > cap) ++bs;
  base = b0;
  return make_int4(bs, (int)((span >> bs) + 1), lo, hi);
}
__device__ __forceinline__ int4 grid_params_of(const double* x, int64_t nb, int64_t cap) {
  if (nb <= 0) return make_int4(0, 0, 0, 0);
  const uint32_t klo = __float_as_uint(f32_rn(x[nb - 1])), khi = __float_as_uint(f32_rn(x[0]));
  int gp = 10;
  while (gp > 0 && (int64_t)((khi >> (23 - gp)) - (klo >> (23 - gp))) + 2 > cap) --gp;
  const int sh = 23 - gp;
  const uint32_t key0 = (klo >> sh) << sh;
  const int cells = (int)((khi - key0) >> sh) + 2;
  return make_int4((int)key0, sh, cells < cap ? cells : (int)cap, (int)khi);  // (as bucket_of)
}

// Phi_k = -(M_k x_k + S_k) over one tile.  The tile's m and x are staged in
// shared memory with coalesced loads; each thread scans its 8 consecutive
// elements (local suffix sums of m x kept in registers), the per-thread
// totals are scanned across the block, and the results leave through shared
// memory with coalesced stores.  kTables: with the orbit step's tables (node
// records, bucket starts, the grid's key shells, their parameters), else Phi
// and, if wanted, M_k.
// Bound with the tables by instruction issue (about 600 a star: three roundings
// to fixed point, two back, a quotient, two fills) and two thirds of the FP64
// pipe; the memory traffic of 76 B a star would take a third of the time.  4 x
// 10^6 stars 154 us, with Phi over M_k in shared memory and 40 registers for
// three blocks an SM (two blocks of 64 registers and no spill: 171).  What the
// tables' readers do not use is not written (float pairs, M_k), neighbours'
// keys and cells come by shuffle, and the tables' parameters are found here by
// two threads of each block while the tile loads (a kernel of one thread per
// segment before took 4.4 us): the stage of 10^7 stars 457 us to 367, of 64 x
// 10^5 stars 328 to 287, of 1021 stars 33 to 20.5.
template <bool kTables>
__global__ void __launch_bounds__(kPotThreads, 3) k_potential(
    Seg S, const int64_t* esc, bool sub, const double* r, const double* x, const double* m,
    const double* tile_m, const double* tile_mx, double* phi, double* Mout, double4_32a* node,
    TableOut T, int lp) {
  pdl_enter();
  extern __shared__ double smem[];
  double* s_m = smem;               // m, then M_k
  double* s_x = smem + kPad8N;      // x
  double* s_p = kTables ? s_m : s_x;  // Phi, over what is not needed any more
  __shared__ double wm[kPotWarps + 1], ws[kPotWarps + 1];
  __shared__ long long wq[kPotWarps], wr[kPotWarps];
  __shared__ int we[kPotWarps];
  const int64_t tile = blockIdx.x >> lp;
  TR R = tile_of(S, esc, tile, sub);
  const int64_t t0 = tile - R.lt;
  const int t = threadIdx.x;
  // this block's part of the tile: elements c0 .. c1 - 1
  const int c0 = (int)(blockIdx.x & ((1u << lp) - 1u)) * (kTile >> lp), c1 = c0 + (kTile >> lp);
  if (R.begin + c0 >= R.end) return;
  // (uniform: the last tile's parts beyond the segment)
  // the tile's loads first, beside the parameters' and the other tiles' sums (the
  // stage of 10^7 stars 359 us with those before, 351 so)
#pragma unroll
  for (int i = 0; i < kPotPer; ++i) {
    const int e = i * kPotThreads + t;
    const int64_t p = R.begin + e;
    const bool ok = p < R.end && p < R.bound_end;
    s_m[pad8(e)] = ok ? m[p] : 0.0;
    s_x[pad8(e)] = ok ? x[p] : 0.0;
  }
  __shared__ int4 s_prm[2];
  __shared__ uint32_t s_base;
  const int64_t nbk = R.bound_end - R.seg_begin;
  if (kTables) {
    const bool out = R.lt == 0 && c0 == 0;  // for the kernels that follow
    if (t == 0) {
      uint32_t base;
      s_prm[0] = bucket_params_of(x + R.seg_begin, nbk, T.boff[R.seg + 1] - T.boff[R.seg] - 1, base);
      s_base = base;
      if (out) {
        T.prm[R.seg] = s_prm[0];
        T.base[R.seg] = base;
      }
    } else if (t == 32) {
      s_prm[1] = grid_params_of(x + R.seg_begin, nbk, T.goff[R.seg + 1] - T.goff[R.seg]);
      if (out) {
        T.gprm[R.seg] = s_prm[1];
        T.gaux[R.seg] = make_float4(0.f, 0.f, __uint_as_float((uint32_t)s_prm[1].x), 0.f);
      }
    }
  }
  // tiles before (M) and after (S) this one, in a fixed order
  double pm = 0.0, ps = 0.0;
  for (int64_t j = t; j < R.nt; j += kPotThreads) {
    if (j < R.lt) pm = pm + tile_m[t0 + j];
    if (j > R.lt) ps = ps + tile_mx[t0 + j];
  }
  block_sums_pot(pm, ps, wm, ws);
  const double Mbefore = pm, Safter = ps;
  __syncthreads();
  const int e0 = t * kPotPer;
  // the tile's sums of m and m x in fixed point (exact inside the tile):
  // the scales from the largest exponents, then the thread's run of 8
  double mx[kPotPer];
  int em = 0, ex = 0;
#pragma unroll
  for (int i = 0; i < kPotPer; ++i) {
    const int q = pad8(e0 + i);
    mx[i] = s_m[q] * s_x[q];
    const int a = exp_of(s_m[q]), b = exp_of(mx[i]);
    em = a > em ? a : em;
    ex = b > ex ? b : ex;
  }
  const int Sm = 49 - (block_max_pot(em, we) - 1023);
  const int Sx = 49 - (block_max_pot(ex, we) - 1023);
  // exclusive suffix of m x along the thread's run, and its total
  long long suf[kPotPer];
  long long ax = 0;
#pragma unroll
  for (int i = kPotPer - 1; i >= 0; --i) {
    suf[i] = ax;
    ax = ax + fix_of(mx[i], Sx);
  }
  long long am = 0;
#pragma unroll
  for (int i = 0; i < kPotPer; ++i) am = am + fix_of(s_m[pad8(e0 + i)], Sm);
  long long pre_m, suf_s;
  block_scans_fix(am, ax, wq, wr, pre_m, suf_s);
  // the part's own elements, and the next one (for the last slope)
  long long run = pre_m;
  const bool own = e0 <= c1 && e0 + kPotPer > c0;
#pragma unroll
  for (int i = 0; i < kPotPer; ++i) {
    if (!own) break;
    const int q = pad8(e0 + i);
    run = run + fix_of(s_m[q], Sm);
    const double Mk = Mbefore + dbl_of_fix(run, Sm);
    const double Sk = Safter + dbl_of_fix(suf_s + suf[i], Sx);
    const double ph = -(Mk * s_x[q] + Sk);
    if (!kTables) s_m[q] = Mk;
    s_p[q] = ph;
  }
  __syncthreads();
  if (!kTables) {
#pragma unroll 4
    for (int e = c0 + t; e < c1; e += kPotThreads) {
      const int64_t p = R.begin + e;
      if (p >= R.end) break;
      const bool bound = p < R.bound_end;
      phi[p] = bound ? s_p[pad8(e)] : 0.0;
      if (Mout) Mout[p] = bound ? s_m[pad8(e)] : 0.0;
    }
    return;
  }
  // Phi, the node records and the orbit step's index tables
  const int c = R.seg;
  const int4 prm = s_prm[0], gpr = s_prm[1];
  const uint32_t base = s_base;
  int* start = T.start + T.boff[c];
  const int64_t cap = T.boff[c + 1] - T.boff[c];
  int* gsh = T.gshell + T.goff[c];
  const int nb = (int)nbk;
  const int lane = t & 31;
#pragma unroll 2
  for (int e = c0 + t; e < c1; e += kPotThreads) {  // (whole warps)
    const int64_t p = R.begin + e;
    const bool bound = p < R.end && p < R.bound_end;
    const int q = pad8(e);
    const double ph = bound ? s_p[q] : 0.0, xk = s_x[q];
    if (p < R.end) {
      phi[p] = ph;
      // the slope of Eq. 6 in 1/r across shell k, (Phi_{k+1} - Phi_k) / (x_k -
      // x_{k+1}) with Phi = 0 at 1/r = 0 beyond the last bound star (the FP64
      // orbit step's shell parameter); a tile's last star, whose neighbour is
      // in the next tile, gets its slope from grid_build
      double w = 0.0;
      if (bound && (p + 1 >= R.bound_end || e + 1 < kTile)) {
        const bool last = p + 1 >= R.bound_end;
        const int q1 = pad8(e + 1 < kTile ? e + 1 : e);
        w = div_rn((last ? 0.0 : s_p[q1]) - ph, xk - (last ? 0.0 : s_x[q1]));
      }
      node[p] = make_double4_32a(xk, ph, r[p], w);
    }
    // the index tables, star by star: bucket starts from the float keys of 1/r
    // of this star and its predecessor, and the grid cells between 1/r of
    // this star and the next (the neighbours' by shuffle)
    const int64_t k = p - R.seg_begin;
    const uint32_t key = __float_as_uint(f32_rn(xk));
    const int cell = grid_last_cell(xk, gpr);
    uint32_t before = __shfl_up_sync(0xFFFFFFFFu, key, 1);
    int after = __shfl_down_sync(0xFFFFFFFFu, cell, 1);
    if (lane == 0)
      before = __float_as_uint(f32_rn(e > 0 ? s_x[pad8(e - 1)] : bound && k > 0 ? x[p - 1] : 0.0));
    if (lane == 31)
      after = grid_last_cell(e + 1 < kTile ? s_x[pad8(e + 1)] : bound && k + 1 < nb ? x[p + 1] : 0.0,
                             gpr);
    bucket_starts_of(0xFFFFFFFFu, bound, (int)k, prm, base, key, before, start, cap);
    grid_shells_of(0xFFFFFFFFu, bound, (int)k, nb, cell, after, gpr, gsh);
  }
  // the ends of both tables, by the part that has their star
  const int64_t ew = prm.w - R.lt * kTile;
  if (nb > 0 && ew >= c0 && ew < c1)
    bucket_close(nb, prm, base, __float_as_uint(f32_rn(s_x[pad8((int)ew)])), start, cap, t,
                 kPotThreads);
  if (nb > 0 && R.lt == 0 && c0 == 0)
    grid_close(grid_last_cell(s_x[0], gpr), gpr, gsh, t, kPotThreads);
}

// ---------------------------------------------------- energy correction
// T' = T + 1/2 [(Phi_new(r_old) - Phi_new(r_new)) - (Phi_old(r_old) -
// Phi_old(r_new))], clamped at 0; both components scaled by sqrt(T'/T).
__global__ void k_correction(Seg S, const int64_t* esc, bool sub, const double* r,
                             const double* x, const double* phi, double* vr, double* vt,
                             const double* r_old, const double* cc, const double* m,
                             int64_t n) {
  pdl_enter();
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  bool active = p < n;
  int c = 0;
  int64_t k = 0, nbc = 0, sb = 0;
  if (active) {
    c = seg_find(S.off, S.n_seg, p);
    sb = S.off[c];
    k = p - sb;
    nbc = nb_eff(S.nb, esc, c, sub);
    active = k < nbc;
  }
  unsigned long long clamp = 0;
  if (active) {
    Table64 T{r + sb, x + sb, phi + sb, nbc};
    double a = vr[p], b = vt[p];
    double Tk = scale_down<1>(a * a + b * b);
    double dnew = phi_of_r(T, r_old[p]) - phi[p];
    double Tp = Tk + scale_down<1>(dnew - cc[p]);
    if (Tp < 0.0) {
      if (m) clamp_energy_add(S.stats, c, m[p], Tp);
      Tp = 0.0;
      clamp = 1;
    }
    if (Tk > 0.0) {
      double f = sqrt_rn(div_rn(Tp, Tk));
      vr[p] = a * f;
      vt[p] = b * f;
    }
  }
  if (clamp) stat_add(S.stats, c, kStClamps, 1ull);
}

// ---------------------------------------------------------- diagnostics
// Both kernels sum runs of 16 consecutive stars per thread and then a tree over
// 256 threads.  512 threads stage the tile with coalesced loads and take the
// stars' terms (products and quotients on the integer pipes); 256 of them sum the
// runs from shared memory (a run of 16 + 1 padded doubles each, free of bank
// conflicts).  Bound by the FP64 pipe (two thirds of the time: the sums) and, at
// 10^6 stars, by the SMs that have two of the 245 tiles; three blocks an SM.
// 42.9 and 46.8 us at 10^6 stars, the masses alone 19.2; with a thread per run
// taking everything, loads of 128 B strides and FP64 divisions, 56.6 and 65.2.
constexpr int kDiagThreads = 512;
constexpr int kDiagPer = kTile / kDiagThreads;
__device__ __forceinline__ int pad16(int e) { return e + (e >> 4); }
constexpr int kPad16N = kTile + kTile / 16;

// block_sum of the first kThreads threads' values in a block of kDiagThreads
__device__ __forceinline__ double diag_sum(double v, double* s) {
  const int t = threadIdx.x;
  if (t < kThreads) s[t] = v;
  __syncthreads();
  for (int w = kThreads / 2; w > 0; w >>= 1) {
    if (t < w) s[t] = s[t] + s[t + w];
    __syncthreads();
  }
  const double r = s[0];
  __syncthreads();
  return r;
}

// kMass: only M_k, the mass up to and including star k, into Mout; else the
// tile's sums of m v^2 and m_k M_{k-1} / r_k.
template <bool kMass>
__global__ void __launch_bounds__(kDiagThreads, 3) k_energy_tiles(Seg S, const double* r,
                                                               const double* vr, const double* vt,
                                                               const double* m,
                                                               const double* tile_m,
                                                               double* tile_k, double* tile_w,
                                                               double* Mout) {
  pdl_enter();
  extern __shared__ double smem[];
  double* s_m = smem;            // m, then the mass inside, then m M / r
  double* s_k = smem + kPad16N;  // m v^2
  __shared__ double s1[kThreads];
  TR R = tile_of(S, nullptr, blockIdx.x, false);
  const int64_t t0 = blockIdx.x - R.lt;
  const int t = threadIdx.x;
#pragma unroll
  for (int j = 0; j < kDiagPer; ++j) {
    const int e = j * kDiagThreads + t;
    const int64_t p = R.begin + e;
    const bool in = p < R.end && p < R.bound_end;
    const double me = in ? m[p] : 0.0;
    s_m[pad16(e)] = me;
    if (!kMass) {
      const double a = in ? vr[p] : 0.0, b = in ? vt[p] : 0.0;
      s_k[pad16(e)] = mul_rn(me, mul_rn(a, a) + mul_rn(b, b));
    }
  }
  double pm = 0.0;
  if (t < kThreads)
    for (int64_t j = t; j < R.lt; j += kThreads) pm = pm + tile_m[t0 + j];
  const double Mbefore = diag_sum(pm, s1);
  if (t < kThreads) {
    double am = 0.0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) am = am + s_m[pad16(t * kPer + i)];
    s1[t] = am;
  }
  __syncthreads();
  // inclusive scan of the runs (fixed shape: doubling steps)
  for (int o = 1; o < kThreads; o <<= 1) {
    const double a = t >= o && t < kThreads ? s1[t - o] : 0.0;
    __syncthreads();
    if (t >= o && t < kThreads) s1[t] = a + s1[t];
    __syncthreads();
  }
  if (t < kThreads) {
    const double base = Mbefore + (t > 0 ? s1[t - 1] : 0.0);
    double run = 0.0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int q = pad16(t * kPer + i);
      const double mi = s_m[q];
      if (!kMass) s_m[q] = base + run;  // the mass strictly inside
      run = run + mi;
      if (kMass) s_m[q] = base + run;
    }
  }
  __syncthreads();
  if (kMass) {
#pragma unroll
    for (int j = 0; j < kDiagPer; ++j) {
      const int e = j * kDiagThreads + t;
      const int64_t p = R.begin + e;
      if (p < R.end) Mout[p] = p < R.bound_end ? s_m[pad16(e)] : 0.0;
    }
    return;
  }
#pragma unroll
  for (int j = 0; j < kDiagPer; ++j) {
    const int e = j * kDiagThreads + t, q = pad16(e);
    const int64_t p = R.begin + e;
    if (p < R.end && p < R.bound_end) s_m[q] = div_rn(mul_rn(m[p], s_m[q]), r[p]);
    else s_m[q] = 0.0;
  }
  __syncthreads();
  double ak = 0.0, aw = 0.0;
  if (t < kThreads) {
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      ak = ak + s_k[pad16(t * kPer + i)];
      aw = aw + s_m[pad16(t * kPer + i)];
    }
  }
  const double tk = diag_sum(ak, s1);
  const double tw = diag_sum(aw, s1);
  if (t == 0) { tile_k[blockIdx.x] = tk; tile_w[blockIdx.x] = tw; }
}

// Core diagnostics (section 4.2, Eq. 19): per bound star k with three
// neighbours on each side, the 6th-order density estimate in the radial
// order, rho_k = (m_{k-2} + ... + m_{k+2}) / (4 pi / 3 (r_{k+3}^3 - r_{k-3}^3));
// per tile the sums of rho, rho^2, rho r and the number of estimates, each
// in a fixed order (runs of 16 per thread, then a fixed tree).
__global__ void __launch_bounds__(kDiagThreads, 3) k_core_tiles(Seg S, const double* r,
                                                             const double* m, double* tile_s1,
                                                             double* tile_s2, double* tile_sr,
                                                             double* tile_n) {
  pdl_enter();
  extern __shared__ double smem[];
  double* s_c = smem;                // r^3 of the tile and 3 stars on each side, then rho
  double* s_m = smem + kPad16N + 8;  // m, likewise, then r
  __shared__ double s[kThreads];
  TR R = tile_of(S, nullptr, blockIdx.x, false);
  const int t = threadIdx.x;
  for (int e = t; e < kTile + 6; e += kDiagThreads) {
    const int64_t p = R.begin + e - 3;
    const bool in = p >= R.seg_begin && p < R.bound_end;
    const double re = in ? r[p] : 0.0;
    s_c[e] = mul_rn(re * re, re);
    s_m[e] = in ? m[p] : 0.0;
  }
  __syncthreads();
  const double c43 = (4.0 * kPi) / 3.0;
  double rho[kDiagPer];
  unsigned ok = 0;
#pragma unroll
  for (int j = 0; j < kDiagPer; ++j) {
    const int e = j * kDiagThreads + t;
    const int64_t p = R.begin + e;
    rho[j] = 0.0;
    if (p >= R.end || p - R.seg_begin < 3 || p + 3 >= R.bound_end) continue;
    const double vol = mul_rn(c43, s_c[e + 6] - s_c[e]);
    if (!pos_num(vol)) continue;
    const double mass = (((s_m[e + 1] + s_m[e + 2]) + s_m[e + 3]) + s_m[e + 4]) + s_m[e + 5];
    rho[j] = div_rn(mass, vol);
    ok |= 1u << j;
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kDiagPer; ++j) {
    const int e = j * kDiagThreads + t;
    s_c[pad16(e)] = rho[j];
    s_m[pad16(e)] = (ok >> j) & 1u ? r[R.begin + e] : 0.0;
  }
  // (an estimate that is not there is a 0 and leaves the sums as they are)
  int count = 0;
#pragma unroll
  for (int j = 0; j < kDiagPer; ++j) count += __syncthreads_count((ok >> j) & 1u);
  double a1 = 0.0, a2 = 0.0, ar = 0.0;
  if (t < kThreads) {
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const double q = s_c[pad16(t * kPer + i)];
      a1 = a1 + q;
      a2 = a2 + mul_rn(q, q);
      ar = ar + mul_rn(q, s_m[pad16(t * kPer + i)]);
    }
  }
  const double t1 = diag_sum(a1, s), t2 = diag_sum(a2, s), tr = diag_sum(ar, s);
  if (t == 0) {
    tile_s1[blockIdx.x] = t1;
    tile_s2[blockIdx.x] = t2;
    tile_sr[blockIdx.x] = tr;
    tile_n[blockIdx.x] = (double)count;
  }
}
constexpr size_t kDiagSmem = sizeof(double) * 2 * (kPad16N + 8);

// The same sums where every cluster has at most kDiagSmall stars: a warp per cluster,
// a run of 16 stars to a lane (the runs, scans and trees above with nothing but
// zeros beyond the warp's), no shared memory and no barriers.  20,000 clusters of
// two stars: sums of the energy 2.3 ms by whole tiles' blocks, 0.07 so, of the core 1.5, 0.03.
constexpr int64_t kDiagSmall = 32 * kPer;
constexpr int kSmallWarps = 8;

__device__ __forceinline__ double warp_tree(double v) {
#pragma unroll
  for (int w = 16; w > 0; w >>= 1) v = v + __shfl_down_sync(0xFFFFFFFFu, v, w);
  return v;
}

template <bool kMass>
__global__ void __launch_bounds__(32 * kSmallWarps) k_energy_small(
    Seg S, int64_t n_tiles, const double* r, const double* vr, const double* vt, const double* m,
    double* tile_k, double* tile_w, double* Mout) {
  pdl_enter();
  const int64_t tile = (int64_t)blockIdx.x * kSmallWarps + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (tile >= n_tiles) return;
  const TR R = tile_of(S, nullptr, tile, false);
  const int64_t p0 = R.begin + lane * kPer;
  auto mass = [&](int64_t p) { return p < R.end && p < R.bound_end ? m[p] : 0.0; };
  double am = 0.0;
  for (int i = 0; i < kPer && p0 + i < R.end; ++i) am = am + mass(p0 + i);
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double a = __shfl_up_sync(0xFFFFFFFFu, am, o);
    if (lane >= o) am = a + am;
  }
  const double below = __shfl_up_sync(0xFFFFFFFFu, am, 1), base = lane > 0 ? below : 0.0;
  double run = 0.0, ak = 0.0, aw = 0.0;
  for (int i = 0; i < kPer && p0 + i < R.end; ++i) {
    const int64_t p = p0 + i;
    const bool in = p < R.bound_end;
    const double mi = in ? m[p] : 0.0, inside = base + run;
    run = run + mi;
    if (kMass) {
      Mout[p] = in ? base + run : 0.0;
    } else if (in) {
      ak = ak + mul_rn(mi, mul_rn(vr[p], vr[p]) + mul_rn(vt[p], vt[p]));
      aw = aw + div_rn(mul_rn(mi, inside), r[p]);
    }
  }
  if (kMass) return;
  const double tk = warp_tree(ak), tw = warp_tree(aw);
  if (lane == 0) {
    tile_k[tile] = tk;
    tile_w[tile] = tw;
  }
}

__global__ void __launch_bounds__(32 * kSmallWarps) k_core_small(Seg S, int64_t n_tiles,
                                                                 const double* r, const double* m,
                                                                 double* tile_s1, double* tile_s2,
                                                                 double* tile_sr, double* tile_n) {
  pdl_enter();
  const int64_t tile = (int64_t)blockIdx.x * kSmallWarps + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (tile >= n_tiles) return;
  const TR R = tile_of(S, nullptr, tile, false);
  const double c43 = (4.0 * kPi) / 3.0;
  double a1 = 0.0, a2 = 0.0, ar = 0.0;
  int count = 0;
  for (int i = 0; i < kPer; ++i) {
    const int64_t p = R.begin + lane * kPer + i;
    if (p + 3 >= R.bound_end) break;
    if (p - R.seg_begin < 3) continue;
    const double ro = r[p + 3], ri = r[p - 3];
    const double vol = mul_rn(c43, mul_rn(ro * ro, ro) - mul_rn(ri * ri, ri));
    if (!pos_num(vol)) continue;
    const double q =
        div_rn((((m[p - 2] + m[p - 1]) + m[p]) + m[p + 1]) + m[p + 2], vol);
    a1 = a1 + q;
    a2 = a2 + mul_rn(q, q);
    ar = ar + mul_rn(q, r[p]);
    ++count;
  }
  const double t1 = warp_tree(a1), t2 = warp_tree(a2), tr = warp_tree(ar);
  count = __reduce_add_sync(0xFFFFFFFFu, count);
  if (lane == 0) {
    tile_s1[tile] = t1;
    tile_s2[tile] = t2;
    tile_sr[tile] = tr;
    tile_n[tile] = (double)count;
  }
}

// per cluster: rho_c = sum rho^2 / sum rho, r_c = sum rho r / sum rho and the
// number of estimates (3 doubles per cluster)
__global__ void __launch_bounds__(kThreads) k_core_final(Seg S, const double* tile_s1,
                                                         const double* tile_s2,
                                                         const double* tile_sr,
                                                         const double* tile_n, double* out3) {
  pdl_enter();
  __shared__ double s[kThreads];
  const int c = blockIdx.x;
  const int64_t t0 = S.tile_off[c], t1 = S.tile_off[c + 1];
  double a1 = 0.0, a2 = 0.0, ar = 0.0, an = 0.0;
  for (int64_t j = t0 + threadIdx.x; j < t1; j += kThreads) {
    a1 = a1 + tile_s1[j];
    a2 = a2 + tile_s2[j];
    ar = ar + tile_sr[j];
    an = an + tile_n[j];
  }
  const double S1 = block_sum(a1, s), S2 = block_sum(a2, s), SR = block_sum(ar, s),
               SN = block_sum(an, s);
  if (threadIdx.x == 0) {
    out3[3 * c + 0] = S1 > 0.0 ? S2 / S1 : 0.0;
    out3[3 * c + 1] = S1 > 0.0 ? SR / S1 : 0.0;
    out3[3 * c + 2] = SN;
  }
}

__global__ void __launch_bounds__(kThreads) k_energy_final(Seg S, const double* tile_k,
                                                           const double* tile_w,
                                                           double* out3) {
  pdl_enter();
  __shared__ double s[kThreads];
  const int c = blockIdx.x;
  int64_t t0 = S.tile_off[c], t1 = S.tile_off[c + 1];
  double ak = 0.0, aw = 0.0;
  for (int64_t j = t0 + threadIdx.x; j < t1; j += kThreads) {
    ak = ak + tile_k[j];
    aw = aw + tile_w[j];
  }
  double K = block_sum(ak, s);
  double W = block_sum(aw, s);
  if (threadIdx.x == 0) {
    out3[3 * c + 0] = 0.5 * K;
    out3[3 * c + 1] = -W;
    out3[3 * c + 2] = 0.5 * K - W;
  }
}

// The first star whose enclosed mass reaches each fraction: a warp per search.  A
// round takes five halvings: lane l (1 to 31) probes node l of the tree of the
// next five midpoints, the answers pick the path (same midpoints and result as
// one halving at a time, which took 13.7 us at 10^6 stars; 8.0).
// (The searches, clusters x fractions, can be more than 2^31: counted in 64 bits,
// the grid strides over those beyond its blocks.)
constexpr int kLagThreads = 128;
__device__ __forceinline__ void lagrange_search(const Seg& S, const double* r, const double* M,
                                                const double* fracs, int nf, double* out,
                                                int64_t i, int lane) {
  const int c = (int)(i / nf), q = (int)(i % nf);
  const int64_t sb = S.off[c], nbc = S.nb[c];
  if (nbc <= 0) {
    if (lane == 0) out[i] = 0.0;
    return;
  }
  const double target = fracs[q] * M[sb + nbc - 1];
  int64_t lo = -1, hi = nbc - 1;  // first k with M_k >= target (M[nb-1] qualifies)
  while (hi - lo > 1) {
    int64_t a = lo, b = hi;
    for (int bit = 30 - __clz(lane | 1); bit >= 0; --bit) {
      if (b - a <= 1) break;
      const int64_t mid = a + ((b - a) >> 1);
      if ((lane >> bit) & 1) b = mid; else a = mid;
    }
    const bool ge = lane > 0 && b - a > 1 && M[sb + a + ((b - a) >> 1)] >= target;
    const unsigned pick = __ballot_sync(0xFFFFFFFFu, ge);
    for (int node = 1; node < 32 && hi - lo > 1;) {
      const int64_t mid = lo + ((hi - lo) >> 1);
      if ((pick >> node) & 1u) {
        hi = mid;
        node = 2 * node + 1;
      } else {
        lo = mid;
        node = 2 * node;
      }
    }
  }
  if (lane == 0) out[i] = r[sb + hi];
}
__global__ void __launch_bounds__(kLagThreads) k_lagrange(Seg S, const double* r, const double* M,
                                                          const double* fracs, int nf,
                                                          double* out) {
  pdl_enter();
  const int64_t n = (int64_t)S.n_seg * nf, step = (int64_t)gridDim.x * (kLagThreads / 32);
  for (int64_t i = (int64_t)blockIdx.x * (kLagThreads / 32) + (threadIdx.x >> 5); i < n; i += step)
    lagrange_search(S, r, M, fracs, nf, out, i, threadIdx.x & 31);
}

__global__ void k_validate(int64_t n, const double* r, const double* vr, const double* vt,
                           const double* m, bool allow_inf, uint32_t* err) {
  pdl_enter();
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  double rr = r[p], a = vr[p], b = vt[p], mm = m[p];
  bool rok = (rr > 0.0) && (isfinite(rr) || (allow_inf && isinf(rr)));
  bool ok = rok && isfinite(a) && isfinite(b) && (b >= 0.0) && isfinite(mm) && (mm >= 0.0);
  if (!ok) set_err(err, kErrInput);
}

// stellar radii or semi-major axes: finite and >= 0 (flag 1 otherwise).  On the
// host, one comparison after the other, a call with 200,003 values took 219 us; 54
// with the copy and the check here.
__global__ void k_check_attr(int64_t n, const double* a, uint32_t* flag) {
  pdl_enter();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const double v = a[p];
  if (!(v >= 0.0) || !lt_inf(v)) *flag = 1u;
}

__global__ void k_check_ids(int64_t n, const int64_t* off, int n_seg, const uint64_t* ids,
                            uint32_t* err) {
  pdl_enter();
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p + 1 >= n) return;
  int c = seg_find(off, n_seg, p);
  if (p + 1 < off[c + 1] && ids[p] == ids[p + 1]) set_err(err, kErrInput);
}

// Whether the staged stars are already in (r, id) order within every
// segment (bit patterns of positive or infinite r order like the values),
// flag bit 0 set otherwise, and the largest id of each segment.
__global__ void k_order_check(int64_t n, const int64_t* off, int n_seg, const double* r,
                              const uint32_t* id, uint32_t* flag, unsigned int* maxid) {
  pdl_enter();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool live = p < n;
  int c = 0;
  uint32_t ip = 0;
  if (live) {
    c = seg_find(off, n_seg, p);
    ip = id[p];
    if (p + 1 < off[c + 1]) {
      const unsigned long long a = ubits(r[p]), b = ubits(r[p + 1]);
      if (!(a < b || (a == b && ip < id[p + 1]))) atomicOr(flag, 1u);
    }
  }
  // one atomic per segment present in the warp
  const unsigned full = __activemask();
  const unsigned peers = __match_any_sync(full, live ? c : -1);
  const unsigned mx = __reduce_max_sync(peers, ip);
  if (live && (threadIdx.x & 31) == __ffs(peers) - 1) atomicMax(maxid + c, mx);
}

// Stars in (r, id) order: duplicate ids by bit bitoff[c] + id of a bitmap (a bit
// found set already is one), and N_bound where the first escaped star (r = inf,
// after all others) or the segment's end is.  Setting a state back at 10^3, 10^5,
// 10^6 stars 127, 145, 258 us with keys, a search of them, reciprocals and a host
// wait between, 110, 134, 230 so.
__global__ void k_place(int64_t n, const int64_t* off, int n_seg, const double* r,
                        const uint32_t* id, const unsigned long long* bitoff,
                        unsigned long long* bitmap, int64_t* nb, uint32_t* err) {
  pdl_enter();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const int c = seg_find(off, n_seg, p);
  const unsigned long long b = bitoff[c] + id[p];
  const unsigned long long bit = 1ull << (b & 63ull);
  if (atomicOr(bitmap + (b >> 6), bit) & bit) set_err(err, kErrInput);
  // the first escaped star's place, or the segment's end (escaped stars last)
  const int64_t sb = off[c];
  const bool gone = ubits(r[p]) >= kInfBits, last = p + 1 == off[c + 1];
  if (gone && (p == sb || ubits(r[p - 1]) < kInfBits)) nb[c] = p - sb;
  if (!gone && last) nb[c] = p + 1 - sb;
}

// one record of the diagnostics ring per segment, after the step end (the
// step counter already advanced): slot (step - 1) mod cap
__global__ void k_diag_ring(Seg S, const double* out3, const uint64_t* dt_last,
                            const double* esc_me, const uint32_t* step, const uint32_t* err,
                            double* ring, int cap) {
  pdl_enter();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= S.n_seg) return;
  const uint32_t stp = *step;
  double* rec = ring + ((size_t)c * cap + (stp - 1u) % (uint32_t)cap) * kDiagFields;
  const double K = out3[3 * c], W = out3[3 * c + 1];
  rec[0] = (double)stp;
  rec[1] = __longlong_as_double((long long)dt_last[c]);
  rec[2] = (double)S.nb[c];
  rec[3] = K;
  rec[4] = W;
  rec[5] = (K + W) + esc_me[2 * c + 1];
  rec[6] = esc_me[2 * c];
  rec[7] = esc_me[2 * c + 1];
  rec[8] = (double)S.stats[(size_t)c * kStStride + kStTrials];
  rec[9] = (double)*err;
}

__global__ void k_nb_from_keys(Seg S, const uint64_t* keys) {
  pdl_enter();
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= S.n_seg) return;
  int64_t sb = S.off[c], se = S.off[c + 1];
  int64_t lo = sb - 1, hi = se;  // first escaper key in [sb, se)
  while (hi - lo > 1) {
    int64_t mid = lo + ((hi - lo) >> 1);
    if (key_is_escaper(keys[mid])) hi = mid; else lo = mid;
  }
  S.nb[c] = hi - sb;
}

__global__ void k_recip(int64_t n, const double* r, double* x) {
  pdl_enter();
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p < n) x[p] = 1.0 / r[p];
}

__global__ void k_make_t32(int64_t n, const double* x, const double* phi, float2* t32) {
  pdl_enter();
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p < n) t32[p] = make_float2((float)x[p], (float)phi[p]);
}

__global__ void k_make_nodes(int64_t n, const double* r, const double* x, const double* phi,
                             const double* M, double4_32a* node) {
  pdl_enter();
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  node[p] = make_double4_32a(x[p], phi[p], r[p], M[p]);
}

__global__ void k_unpack_orbit(int64_t n, const RecA* ra, const RecB* rb, double* r_new,
                               double* vr_new, double* vt_new) {
  pdl_enter();
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  r_new[p] = ra[p].r;
  if (vr_new) vr_new[p] = rb[p].vr;
  if (vt_new) vt_new[p] = rb[p].vt;
}

inline unsigned blocks_for(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

// the first words of a Carve's block from its image, zero up to `words`
struct CarveImage {
  uint4 w[128];
};
__global__ void k_carve(uint4* dst, int64_t words, int image, CarveImage im) {
  pdl_enter();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < words) dst[i] = i < image ? im.w[i] : make_uint4(0u, 0u, 0u, 0u);
}

}  // namespace

void launch_nb_from_keys(const SegLayout& L, const uint64_t* keys, cudaStream_t st) {
  launch_k(k_nb_from_keys, blocks_for(L.n_seg, 128), 128, 0, st, L.dev(), keys);
}

void launch_recip(int64_t n, const double* r, double* x, cudaStream_t st) {
  if (n > 0) launch_k(k_recip, blocks_for(n, 256), 256, 0, st, n, r, x);
}

void launch_make_t32(int64_t n, const double* x, const double* phi, float2* t32,
                     cudaStream_t st) {
  if (n > 0) launch_k(k_make_t32, blocks_for(n, 256), 256, 0, st, n, x, phi, t32);
}

void launch_make_nodes(int64_t n, const double* r, const double* x, const double* phi,
                       const double* M, double4_32a* node, cudaStream_t st) {
  if (n > 0) launch_k(k_make_nodes, blocks_for(n, 256), 256, 0, st, n, r, x, phi, M, node);
}

void launch_unpack_orbit(int64_t n, const RecA* ra, const RecB* rb, double* r_new,
                         double* vr_new, double* vt_new, cudaStream_t st) {
  if (n > 0)
    launch_k(k_unpack_orbit, blocks_for(n, 256), 256, 0, st, n, ra, rb, r_new, vr_new, vt_new);
}

// ------------------------------------------------------------------ host
void Carve::copy(unsigned char* to, const void* from, size_t n) { memcpy(to, from, n); }

cudaError_t Carve::alloc(void*& block, cudaStream_t st) {
  cudaError_t e = cudaMallocAsync(&block, bytes_ ? bytes_ : 1, st);
  if (e) {
    block = nullptr;
    return e;
  }
  for (const Part& q : parts_) *q.ptr = (unsigned char*)block + q.at;
  if (zero_ == 0) return cudaSuccess;
  if (image_.size() <= sizeof(CarveImage)) {
    CarveImage im;
    memset(&im, 0, sizeof(im));
    if (!image_.empty()) memcpy(&im, image_.data(), image_.size());
    const int64_t words = (int64_t)(zero_ / 16);
    launch_k(k_carve, blocks_for(words, 256), 256, 0, st, (uint4*)block, words,
             (int)(image_.size() / 16), im);
    e = cudaGetLastError();
  } else {
    e = cudaMemcpyAsync(block, image_.data(), image_.size(), cudaMemcpyHostToDevice, st);
    if (!e && zero_ > image_.size())
      e = cudaMemsetAsync((unsigned char*)block + image_.size(), 0, zero_ - image_.size(), st);
    if (!e) e = cudaStreamSynchronize(st);  // the image lives on the caller's stack
  }
  if (e) {
    cudaFreeAsync(block, st);
    block = nullptr;
  }
  return e;
}

cudaError_t alloc_layout(SegLayout& L, const std::vector<int64_t>& sizes,
                         const std::vector<uint64_t>& seeds, const std::vector<double>& lnL,
                         int bin_size, cudaStream_t st) {
  L.n_seg = (int)sizes.size();
  L.bin_size = bin_size;
  L.h_off.assign(L.n_seg + 1, 0);
  L.h_tile_off.assign(L.n_seg + 1, 0);
  L.h_pair_off.assign(L.n_seg + 1, 0);
  L.h_bin_off.assign(L.n_seg + 1, 0);
  L.max_seg = 0;
  for (int c = 0; c < L.n_seg; ++c) {
    int64_t nc = sizes[c];
    int64_t nt = (nc + kTile - 1) / kTile;
    L.h_off[c + 1] = L.h_off[c] + nc;
    L.h_tile_off[c + 1] = L.h_tile_off[c] + nt;
    L.h_pair_off[c + 1] = L.h_pair_off[c] + nc / 2;
    L.h_bin_off[c + 1] = L.h_bin_off[c] + (nc + bin_size - 1) / bin_size;
    if (nc > L.max_seg) L.max_seg = nc;
  }
  L.n = L.h_off[L.n_seg];
  L.n_tiles = L.h_tile_off[L.n_seg];
  L.n_pairs = L.h_pair_off[L.n_seg];
  L.n_bins = L.h_bin_off[L.n_seg];
  const size_t seg = (size_t)L.n_seg, s1 = seg + 1;
  const std::vector<uint64_t> inf(seg, 0x7FF0000000000000ull);
  Carve C;
  C.put(L.off, L.h_off.data(), s1);
  C.put(L.tile_off, L.h_tile_off.data(), s1);
  C.put(L.pair_off, L.h_pair_off.data(), s1);
  C.put(L.bin_off, L.h_bin_off.data(), s1);
  C.put(L.seed, seeds.data(), seg);
  C.put(L.lnL, lnL.data(), seg);
  C.put(L.nb, sizes.data(), seg);
  C.put(L.dt_bits, inf.data(), seg);
  C.put(L.dt_last, inf.data(), seg);
  C.zero(L.esc_step, seg);
  C.zero(L.stats, kStStride * seg);
  C.zero(L.esc_me, 2 * seg);
  C.zero(L.dt_cap, seg);
  C.zero(L.tile_done, (size_t)L.n_tiles + 1);
  return C.alloc(L.block, st);
}

void free_layout(SegLayout& L, cudaStream_t st) {
  if (L.block) cudaFreeAsync(L.block, st);
  L = SegLayout();
}

void launch_make_keys(const SegLayout& L, const double* r, const uint32_t* id, uint64_t* keys,
                      cudaStream_t st) {
  if (L.n) launch_k(k_make_keys, blocks_for(L.n, 256), 256, 0, st, L.n, r, id, keys);
}

void launch_make_records(const SegLayout& L, const double* r, const double* vr,
                         const double* vt, const double* m, const uint32_t* id, RecA* ra,
                         RecB* rb, cudaStream_t st) {
  if (L.n)
    launch_k(k_make_records, blocks_for(L.n, 256), 256, 0, st, L.n, r, vr, vt, m, id, ra, rb);
}

void launch_id_keys(const SegLayout& L, const uint32_t* id, uint64_t* keys, cudaStream_t st) {
  if (L.n) launch_k(k_id_keys, blocks_for(L.n, 256), 256, 0, st, L.n, id, keys);
}

void launch_rekey_radius(const SegLayout& L, const uint32_t* perm, const double* r,
                         const uint32_t* id, uint64_t* keys, cudaStream_t st) {
  if (L.n) launch_k(k_rekey_radius, blocks_for(L.n, 256), 256, 0, st, L.n, perm, r, id, keys);
}

void launch_gather(const SegLayout& L, const uint32_t* perm, const RecA* ra, const RecB* rb,
                   double* r, double* x, double* vr, double* vt, double* m, uint32_t* id,
                   cudaStream_t st) {
  if (L.n)
    launch_k(k_gather, blocks_for(L.n, 256), 256, 0, st, L.n, perm, ra, rb, r, x, vr, vt, m, id);
}

void launch_gather_step(const SegLayout& L, BinWork* B, const uint32_t* order_in,
                        const RecA* ra, const RecB* rb, const double* r_in, double* r_out,
                        double* x_out, double* m, uint32_t* id, uint32_t* order_out,
                        double* r_old, double* c, double* tile_m, double* tile_mx,
                        const double* Rp, double* Rout, const double* Ap, double* Aout,
                        bool exact, cudaStream_t st) {
  if (!L.n_tiles) return;
  GatherOut O;
  O.r = r_out; O.x = x_out; O.m = m;
  O.id = id; O.order = order_out;
  O.r_old = r_old; O.c = c;
  O.tile_m = tile_m; O.tile_mx = tile_mx;
  O.Rp = Rp; O.Ap = Ap;
  O.R = Rout; O.A = Aout;
  constexpr int kPart = kGatSpan + 2 * kRunMax;  // threads
  const bool part = L.n_tiles <= kGatPartTiles, few = L.n_tiles <= kGatFewTiles;
  launch_k(exact ? (part  ? k_gather_step<true, kGatSpan, kPart>
                    : few ? k_gather_step<true, kTile, 1024>
                          : k_gather_step<true, kTile, 512>)
                 : (part  ? k_gather_step<false, kGatSpan, kPart>
                    : few ? k_gather_step<false, kTile, 1024>
                          : k_gather_step<false, kTile, 512>),
           (unsigned)(part ? L.n_tiles * (kTile / kGatSpan) : L.n_tiles),
           part ? kPart : few ? 1024 : 512, 0, st, L.dev(), L.esc_step, L.n, order_in, ra, rb, r_in,
           O, B ? B->cnt : nullptr, B ? B->n_bins : 0, B ? B->desc : nullptr, B ? B->n_tiles : 0,
           B ? B->ctl : nullptr, L.tile_done);
}

void launch_phi_old(const SegLayout& L, const double* r_in, const double* x_in, const double* r,
                    const double* x, const double* phi, const double4_32a* node, RecB* rb,
                    bool div_form, cudaStream_t st, const GridBuild* grid) {
  if (!L.n_tiles) return;
  const int per = L.n_tiles <= kPoFewTiles ? 1 : kPoPer;
  const unsigned gb =
      grid ? (unsigned)((grid->total + grid->n_tiles + kPoThreads - 1) / kPoThreads) : 0u;
  launch_k(per == 1 ? (div_form ? k_phi_old<true, 1> : k_phi_old<false, 1>)
                    : (div_form ? k_phi_old<true, kPoPer> : k_phi_old<false, kPoPer>),
           gb + (unsigned)(L.n_tiles * (kTile / (kPoThreads * per))), kPoThreads, 0, st, L.dev(),
           L.esc_step, r_in, x_in, r, x, phi, node, rb, grid ? *grid : GridBuild(), gb);
}

void launch_velocities(const SegLayout& L, const uint32_t* order, const RecB* rb,
                       const double* phi, const double* m, double* vr, double* vt, bool correct,
                       const double* r_old, const double* c, uint32_t* step, cudaStream_t st) {
  if (!L.n_seg) return;
  StepEnd E;
  E.esc = L.esc_step;
  E.dt_last = L.dt_last;
  E.step = step;
  E.r_old = r_old;
  E.e = c;
  E.esc_me = L.esc_me;
  uint32_t* done = L.tile_done + L.n_tiles;
  const auto kernel = correct ? k_velocities<true> : k_velocities<false>;
  // Many blocks: the step's end after them.  In the same launch it saves the next
  // one's 3 us, but every block waits for its turn at the counter: potential,
  // correction and end of 10^5, 4 x 10^5, 10^6, 2 x 10^6, 10^7 stars 45.7, 72.4, 117.5,
  // 205.6, 805 us in one launch, 48.5, 75.9, 117.9, 202.1, 782 in two.
  const bool together = L.n <= kEndWithVelocities;
  E.done = together ? done : nullptr;
  launch_k(kernel, (unsigned)(together ? L.n_seg : 0) + blocks_for(L.n, 256), 256, 0, st, L.dev(),
           L.n, order, rb, phi, m, vr, vt, E);
  if (together) return;
  E.done = done;
  launch_k(kernel, (unsigned)L.n_seg, 256, 0, st, L.dev(), (int64_t)0, order, rb, phi, m, vr, vt, E);
}

constexpr size_t kPotentialSmem = sizeof(double) * 2 * kPad8N;

template <int kKind>
void tile_sums_prepare() {
  cudaFuncSetAttribute(k_tile_sums<kKind>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)(sizeof(double) * kTile * 2));
}

void diag_prepare() {
  cudaFuncSetAttribute(k_energy_tiles<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)kDiagSmem);
  cudaFuncSetAttribute(k_energy_tiles<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)kDiagSmem);
  cudaFuncSetAttribute(k_core_tiles, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDiagSmem);
}

void potential_prepare() {
  cudaFuncSetAttribute(k_potential<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)kPotentialSmem);
  cudaFuncSetAttribute(k_potential<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)kPotentialSmem);
  tile_sums_prepare<kSumsOfX>();
  tile_sums_prepare<kSumsRecip>();
}


void launch_potential(const SegLayout& L, const double* r, const double* x, const double* m,
                      double* tile_m, double* tile_mx, double* phi, double* Mout, bool nb_sub,
                      cudaStream_t st, bool sums_ready, double4_32a* node,
                      const TableOut* tables, double* recip, bool over_m) {
  if (!L.n_tiles) return;
  Seg S = L.dev();
  if (recip)
    launch_tile_sums<kSumsRecip>(L, nb_sub, r, m, tile_m, tile_mx, recip, st);
  else if (!sums_ready)
    launch_tile_sums<kSumsOfX>(L, nb_sub, x, m, tile_m, tile_mx, nullptr, st);
  int lp = 0;
  while (!over_m && lp < kPotParts && L.n_tiles << (lp + 1) <= kPotBlocks) ++lp;
  launch_k(tables ? k_potential<true> : k_potential<false>, (unsigned)(L.n_tiles << lp),
           kPotThreads, kPotentialSmem, st, S, L.esc_step, nb_sub, r, x, m, tile_m, tile_mx, phi,
           Mout, node, tables ? *tables : TableOut(), lp);
}

void launch_correction(const SegLayout& L, const double* r, const double* x,
                       const double* phi, double* vr, double* vt, const double* r_old,
                       const double* c, bool nb_sub, uint32_t* err, cudaStream_t st,
                       const double* m) {
  (void)err;
  if (!L.n) return;
  launch_k(k_correction, blocks_for(L.n, 128), 128, 0, st, L.dev(), L.esc_step, nb_sub, r, x, phi,
                                                    vr, vt, r_old, c, m, L.n);
}

void launch_energy(const SegLayout& L, const double* r, const double* vr, const double* vt,
                   const double* m, double* tile_m, double* tile_k, double* tile_w,
                   double* out3, cudaStream_t st) {
  if (!L.n_tiles) return;
  Seg S = L.dev();
  if (L.max_seg <= kDiagSmall) {
    launch_k(k_energy_small<false>, blocks_for(L.n_tiles, kSmallWarps), 32 * kSmallWarps, 0, st, S,
             L.n_tiles, r, vr, vt, m, tile_k, tile_w, nullptr);
  } else {
    launch_tile_sums<kSumsMass>(L, false, nullptr, m, tile_m, nullptr, nullptr, st);
    launch_k(k_energy_tiles<false>, (unsigned)L.n_tiles, kDiagThreads, kDiagSmem, st, S, r, vr, vt,
             m, tile_m, tile_k, tile_w, nullptr);
  }
  launch_k(k_energy_final, (unsigned)L.n_seg, kThreads, 0, st, S, tile_k, tile_w, out3);
}

int energy_kernels(const SegLayout& L) { return L.max_seg <= kDiagSmall ? 2 : 3; }

void launch_masses(const SegLayout& L, const double* m, double* tile_m, double* Mout,
                   cudaStream_t st) {
  if (!L.n_tiles) return;
  Seg S = L.dev();
  if (L.max_seg <= kDiagSmall) {
    launch_k(k_energy_small<true>, blocks_for(L.n_tiles, kSmallWarps), 32 * kSmallWarps, 0, st, S,
             L.n_tiles, nullptr, nullptr, nullptr, m, nullptr, nullptr, Mout);
    return;
  }
  launch_tile_sums<kSumsMass>(L, false, nullptr, m, tile_m, nullptr, nullptr, st);
  launch_k(k_energy_tiles<true>, (unsigned)L.n_tiles, kDiagThreads, kDiagSmem, st, S, nullptr,
           nullptr, nullptr, m, tile_m, nullptr, nullptr, Mout);
}

void launch_diag_ring(const SegLayout& L, const double* out3, const uint32_t* step,
                      const uint32_t* err, double* ring, int cap, cudaStream_t st) {
  if (!L.n_seg || cap <= 0) return;
  launch_k(k_diag_ring, (unsigned)((L.n_seg + 127) / 128), 128, 0, st, L.dev(), out3, L.dt_last,
                                                                L.esc_me, step, err, ring, cap);
}

void launch_core(const SegLayout& L, const double* r, const double* m, double* tiles4,
                 double* out3, cudaStream_t st) {
  if (!L.n_tiles) return;
  Seg S = L.dev();
  const int64_t t = L.n_tiles;
  if (L.max_seg <= kDiagSmall)
    launch_k(k_core_small, blocks_for(t, kSmallWarps), 32 * kSmallWarps, 0, st, S, t, r, m, tiles4,
             tiles4 + t, tiles4 + 2 * t, tiles4 + 3 * t);
  else
    launch_k(k_core_tiles, (unsigned)t, kDiagThreads, kDiagSmem, st, S, r, m, tiles4, tiles4 + t,
             tiles4 + 2 * t, tiles4 + 3 * t);
  launch_k(k_core_final, (unsigned)L.n_seg, kThreads, 0, st, S, tiles4, tiles4 + t, tiles4 + 2 * t,
                                                       tiles4 + 3 * t, out3);
}

void launch_lagrange(const SegLayout& L, const double* r, const double* M,
                     const double* fracs, int nf, double* out, cudaStream_t st) {
  const int64_t n = (int64_t)L.n_seg * nf;
  const int64_t blocks = (n + kLagThreads / 32 - 1) / (kLagThreads / 32), most = 1 << 24;
  if (n)
    launch_k(k_lagrange, (unsigned)(blocks < most ? blocks : most), kLagThreads, 0, st, L.dev(), r,
             M, fracs, nf, out);
}

void launch_validate(const SegLayout& L, const double* r, const double* vr,
                     const double* vt, const double* m, bool allow_inf, uint32_t* err,
                     cudaStream_t st) {
  if (L.n) launch_k(k_validate, blocks_for(L.n, 256), 256, 0, st, L.n, r, vr, vt, m, allow_inf, err);
}

void launch_order_check(const SegLayout& L, const double* r, const uint32_t* id, uint32_t* flag,
                        unsigned int* maxid, cudaStream_t st) {
  if (L.n) launch_k(k_order_check, blocks_for(L.n, 256), 256, 0, st, L.n, L.off, L.n_seg, r, id, flag,
                                                               maxid);
}

void launch_place(const SegLayout& L, const double* r, const uint32_t* id,
                  const unsigned long long* bitoff, unsigned long long* bitmap, uint32_t* err,
                  cudaStream_t st) {
  if (L.n)
    launch_k(k_place, blocks_for(L.n, 256), 256, 0, st, L.n, L.off, L.n_seg, r, id, bitoff, bitmap,
             L.nb, err);
}

void launch_check_attr(int64_t n, const double* a, uint32_t* flag, cudaStream_t st) {
  if (n > 0) launch_k(k_check_attr, blocks_for(n, 256), 256, 0, st, n, a, flag);
}

void launch_check_ids(const SegLayout& L, const uint64_t* sorted_ids, uint32_t* err,
                      cudaStream_t st) {
  if (L.n > 1)
    launch_k(k_check_ids, blocks_for(L.n, 256), 256, 0, st, L.n, L.off, L.n_seg, sorted_ids, err);
}

CMC_DEBUG_SITE_ACCESSOR

}  // namespace cmc
