// Sort of the stars by radius (section 2.1 step 6).
//
// The timestep sorts by counting, on the shells of the old table (see BinWork
// and k_bin_scan below).  States in no particular order, the stage call and
// timesteps configured so take the radix sort:
//
// A stable least-significant-digit radix sort over 8-bit digits of the
// 64-bit key, run independently inside every segment (cluster) of the
// state.  Each digit pass is a single "onesweep" kernel: a CTA takes the
// next tile by atomic ticket, ranks its keys with a stable warp-level
// multisplit, publishes its digit counts, and obtains the counts of all
// earlier tiles of its segment by decoupled look-back on those published
// words (integer sums, so the result does not depend on timing).  Tiles are
// taken in ticket order, so every tile a CTA waits on is already running;
// each wait is still bounded and reports a timeout instead of spinning
// forever.  The tile is reordered in shared memory so that the scatter
// writes contiguous runs.
//
// Two shape parameters are chosen at initialisation by timing them on the
// real keys, where the timestep uses them: keys per thread (8 or 16, so tiles
// of 2048 or 4096) and the multisplit (one __match_any_sync per key, or nine
// __ballot_sync intersected bit by bit).
#include <utility>
#include <vector>

#include "cmc_host.hpp"

namespace cmc {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr unsigned long long kFlagAgg = 1ull << 62;
constexpr unsigned long long kFlagInc = 2ull << 62;
constexpr unsigned long long kCountMask = (1ull << 62) - 1;
// Bounds of the device waits, in the library's device memory so that a
// change reaches kernels already captured in a graph: polls of a look-back
// word before a tile gives up on it (and reports a timeout), and moves of
// the tie fix's insertion sort before it gives up on a run.
constexpr int kSpinCapDefault = 1 << 22;
constexpr long long kTieMoveCapDefault = 1ll << 22;
__device__ int g_spin_cap = kSpinCapDefault;
__device__ long long g_tie_move_cap = kTieMoveCapDefault;
constexpr int kMaxPasses = 8;
static_assert(kThreads == kBins, "one thread per digit");

__device__ __forceinline__ unsigned lanemask_lt() {
  unsigned m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

__device__ __forceinline__ unsigned long long ld_volatile(const unsigned long long* p) {
  return *(volatile const unsigned long long*)p;
}

struct TileRange {
  int seg;
  int64_t lt;        // tile index inside the segment
  int64_t seg_begin, begin, end;
};

__device__ __forceinline__ TileRange tile_range(const int64_t* off, const int64_t* tile_off,
                                                int n_seg, int64_t t, int tile) {
  TileRange R;
  R.seg = seg_find(tile_off, n_seg, t);
  R.lt = t - tile_off[R.seg];
  R.seg_begin = off[R.seg];
  R.begin = R.seg_begin + R.lt * tile;
  int64_t se = off[R.seg + 1];
  R.end = R.begin + tile < se ? R.begin + tile : se;
  return R;
}

// block-wide exclusive scan of one value per thread (256 threads)
__device__ __forceinline__ uint32_t block_excl_scan_u32(uint32_t v, uint32_t* s_warp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[warp] = x;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < kWarps ? s_warp[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < kWarps) s_warp[lane] = w;
  }
  __syncthreads();
  uint32_t before = warp ? s_warp[warp - 1] : 0;
  return before + x - v;
}

// ---------------------------------------------------------------- upsweep
// Per-segment histogram of every pass digit over tiles of kTile keys.  Each
// warp counts into its own shared-memory histogram (collisions only among
// its 32 lanes); the warps' histograms are summed before one global atomic
// per bin.  The last block of a segment to finish (a counter per segment,
// no waiting) turns that segment's histograms into exclusive scans.
__global__ void __launch_bounds__(kThreads) k_upsweep(const int64_t* off, const int64_t* tile_off,
                                                      int n_seg, const uint64_t* keys,
                                                      int first_pass, int passes,
                                                      uint32_t* hist, uint32_t* done) {
  pdl_enter();
  __shared__ uint32_t s_warp[kWarps];
  __shared__ bool s_last;
  extern __shared__ uint32_t h[];  // [kWarps][passes][kBins]
  const int warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < kWarps * passes * kBins; i += kThreads) h[i] = 0;
  __syncthreads();
  TileRange R = tile_range(off, tile_off, n_seg, blockIdx.x, kTile);
  uint32_t* hw = h + (size_t)warp * passes * kBins;
  for (int64_t p = R.begin + threadIdx.x; p < R.end; p += kThreads) {
    const uint64_t k = keys[p];
    for (int q = 0; q < passes; ++q)
      atomicAdd(&hw[q * kBins + (int)((k >> (8 * (first_pass + q))) & 0xFF)], 1u);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < passes * kBins; i += kThreads) {
    uint32_t s = 0;
    for (int w = 0; w < kWarps; ++w) s += h[(size_t)w * passes * kBins + i];
    if (s) atomicAdd(&hist[((size_t)R.seg * passes) * kBins + i], s);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();  // this block's counts before its arrival
    const uint32_t tiles = (uint32_t)(tile_off[R.seg + 1] - tile_off[R.seg]);
    s_last = atomicAdd(&done[R.seg], 1u) == tiles - 1u;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();  // every block's counts, read past L1
  for (int q = 0; q < passes; ++q) {
    uint32_t* hq = hist + ((size_t)R.seg * passes + q) * kBins;
    const uint32_t v = __ldcg(hq + threadIdx.x);
    const uint32_t e = block_excl_scan_u32(v, s_warp);
    hq[threadIdx.x] = e;
    __syncthreads();  // s_warp is read by the scan's last step
  }
}

template <int IPT>
struct PassSmem {
  uint64_t key[kThreads * IPT];
  uint32_t val[kThreads * IPT];
  uint32_t whist[kWarps][kBins];
  int64_t gbase[kBins];
  uint32_t dstart[kBins];
  uint32_t s_warp[kWarps];
  int64_t tile;
};

// lanes of the warp that hold the same digit (digits 0..256, 256 = no key),
// from one ballot per digit bit
__device__ __forceinline__ unsigned peers_ballot(int d) {
  unsigned m = 0xffffffffu;
#pragma unroll
  for (int b = 0; b < 9; ++b) {
    const bool bit = (d >> b) & 1;
    const unsigned x = __ballot_sync(0xffffffffu, bit);
    m &= bit ? x : ~x;
  }
  return m;
}

constexpr int kRankMatch = 0;   // __match_any_sync
constexpr int kRankBallot = 1;  // nine __ballot_sync

// ------------------------------------------------------------- onesweep
template <bool kValIdentity, int IPT, int kRank>
__global__ void __launch_bounds__(kThreads, (IPT <= 8 ? 6 : 3))
    k_pass(const int64_t* off, const int64_t* tile_off, int n_seg, int64_t n_tiles,
           const uint64_t* keys_in, const uint32_t* vals_in,
           uint64_t* keys_out, uint32_t* vals_out, int pass, int q,
           int passes, const uint32_t* base, unsigned long long* desc, uint32_t* tickets,
           uint32_t* err) {
  pdl_enter();
  constexpr int kTileKeys = kThreads * IPT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PassSmem<IPT>& S = *reinterpret_cast<PassSmem<IPT>*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int shift = 8 * pass;

  if (tid == 0) S.tile = (int64_t)atomicAdd(tickets + q, 1u);
  for (int i = tid; i < kWarps * kBins; i += kThreads) (&S.whist[0][0])[i] = 0;
  __syncthreads();
  const int64_t t = S.tile;
  TileRange R = tile_range(off, tile_off, n_seg, t, kTileKeys);
  const int64_t n_items = R.end - R.begin;

  // warp-striped load: warp w owns elements [w*32*IPT, (w+1)*32*IPT)
  uint64_t k[IPT];
  uint32_t v[IPT];
  int dg[IPT];
#pragma unroll
  for (int i = 0; i < IPT; ++i) {
    int64_t e = (int64_t)warp * (32 * IPT) + i * 32 + lane;
    int64_t p = R.begin + e;
    bool valid = e < n_items;
    k[i] = valid ? keys_in[p] : 0ull;
    v[i] = valid ? (kValIdentity ? (uint32_t)p : vals_in[p]) : 0u;
    dg[i] = valid ? (int)((k[i] >> shift) & 0xFF) : kBins;
  }

  // warp-level multisplit ranks (stable: slot order, then lane order).
  // The leader of each group of equal digits adds the group's size to the
  // warp's counter with a shared-memory atomic; the counts before (the
  // atomics' results) are read only after a group of slots has been
  // issued, so the round trips overlap.  A __syncwarp between slots orders
  // the updates of one counter by different leaders in slot order.
  uint32_t rank[IPT];
  const unsigned lt_mask = lanemask_lt();
  constexpr int kGrp = IPT < 4 ? IPT : 4;
#pragma unroll
  for (int i0 = 0; i0 < IPT; i0 += kGrp) {
    unsigned pe[kGrp];
    uint32_t old[kGrp];
#pragma unroll
    for (int j = 0; j < kGrp; ++j) {
      const int i = i0 + j;
      pe[j] = kRank == kRankMatch ? __match_any_sync(0xffffffffu, dg[i]) : peers_ballot(dg[i]);
      old[j] = 0;
      if (lane == __ffs(pe[j]) - 1 && dg[i] < kBins)
        old[j] = atomicAdd(&S.whist[warp][dg[i]], (uint32_t)__popc(pe[j]));
      __syncwarp();
    }
#pragma unroll
    for (int j = 0; j < kGrp; ++j) {
      const uint32_t o = __shfl_sync(0xffffffffu, old[j], __ffs(pe[j]) - 1);
      rank[i0 + j] = o + __popc(pe[j] & lt_mask);
    }
  }
  __syncthreads();

  // per digit: exclusive prefix over warps, tile count
  const int d = tid;
  uint32_t cnt = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    uint32_t c = S.whist[w][d];
    S.whist[w][d] = cnt;
    cnt += c;
  }

  // decoupled look-back over the earlier tiles of this segment
  unsigned long long* my = desc + ((size_t)q * n_tiles + t) * kBins + d;
  uint64_t excl = 0;
  if (R.lt == 0) {
    atomicExch(my, kFlagInc | (unsigned long long)cnt);
  } else {
    atomicExch(my, kFlagAgg | (unsigned long long)cnt);
    int64_t j = t - 1;
    const int64_t first = t - R.lt;
    const int spin_cap = g_spin_cap;
    int spins = 0;
    while (j >= first) {
      unsigned long long w = ld_volatile(desc + ((size_t)q * n_tiles + j) * kBins + d);
      if ((w & ~kCountMask) == 0) {
        if (++spins > spin_cap) {
          set_err(err, kErrTimeout);
          --j;
          spins = 0;
          continue;
        }
        if (spins > 32) __nanosleep(64);
        continue;
      }
      excl += (w & kCountMask);
      if ((w & ~kCountMask) == kFlagInc) break;
      --j;
    }
    atomicExch(my, kFlagInc | (unsigned long long)(excl + cnt));
  }

  uint32_t ds = block_excl_scan_u32(cnt, S.s_warp);
  S.dstart[d] = ds;
  S.gbase[d] = R.seg_begin + (int64_t)base[((size_t)R.seg * passes + q) * kBins + d] +
               (int64_t)excl - (int64_t)ds;
  __syncthreads();

  // reorder the tile in shared memory by digit
#pragma unroll
  for (int i = 0; i < IPT; ++i) {
    if (dg[i] < kBins) {
      uint32_t lp = S.dstart[dg[i]] + S.whist[warp][dg[i]] + rank[i];
      S.key[lp] = k[i];
      S.val[lp] = v[i];
    }
  }
  __syncthreads();

  // contiguous runs per digit go out coalesced; a destination outside the
  // segment (possible only after a timed-out look-back) is dropped
  const int64_t seg_end = off[R.seg + 1];
  for (int lp = tid; lp < n_items; lp += kThreads) {
    uint64_t kk = S.key[lp];
    int dd = (int)((kk >> shift) & 0xFF);
    int64_t dest = S.gbase[dd] + lp;
    if (dest < R.seg_begin || dest >= seg_end) {
      set_err(err, kErrTimeout);
      continue;
    }
    keys_out[dest] = kk;
    vals_out[dest] = S.val[lp];
  }
}

// ------------------------------------------------------------- tie fix
// Runs of keys equal in their bits above `shift` are put in (key, id) order
// (insertion sort by one thread per run; a run that is already ordered
// costs one pass): finite radii in (r, id) order, escapers in id order.

__global__ void k_tiefix(const int64_t* off, int n_seg, int64_t n, uint64_t* keys,
                         uint32_t* vals, const uint32_t* ids_by_val, int id_stride, int shift,
                         uint32_t* err, unsigned long long* stats) {
  pdl_enter();
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  if (*err & kErrTimeout) {
    vals[p] = (uint32_t)p;  // as k_long_runs: no order that was not written
    return;
  }
  int c = seg_find(off, n_seg, p);
  int64_t sb = off[c], se = off[c + 1];
  const uint64_t kp = keys[p], hp = kp >> shift;
  if (p + 1 >= se || (keys[p + 1] >> shift) != hp) return;
  if (p > sb && (keys[p - 1] >> shift) == hp) return;  // not the start of the run
  int64_t e = p + 2;
  while (e < se && (keys[e] >> shift) == hp) ++e;
  // insertion sort of the run by (key, id)
  const long long move_cap = g_tie_move_cap;
  long long moves = 0;
  for (int64_t i = p + 1; i < e; ++i) {
    const uint64_t kv = keys[i];
    const uint32_t v = vals[i];
    const uint32_t idv = ids_by_val[(size_t)v * id_stride];
    int64_t j = i - 1;
    while (j >= p) {
      const uint64_t kj = keys[j];
      if (!(kj > kv || (kj == kv && ids_by_val[(size_t)vals[j] * id_stride] > idv))) break;
      keys[j + 1] = kj;
      vals[j + 1] = vals[j];
      --j;
      if (++moves > move_cap) {
        set_err(err, kErrTies);
        keys[j + 1] = kv;
        vals[j + 1] = v;
        return;
      }
    }
    keys[j + 1] = kv;
    vals[j + 1] = v;
  }
  // the run's groups of equal radii, each counted at its second star (as the
  // timestep's gather does; escapers have keys of their own)
  unsigned long long groups = 0;
  for (int64_t i = p + 1; i < e; ++i)
    groups += keys[i] == keys[i - 1] && (i - 1 == p || keys[i - 2] != keys[i]);
  if (groups && stats) atomicAdd(stats + (size_t)c * kStStride + kStTies, groups);
}

// ------------------------------------------------------- counting sort
// (see BinWork).  At N = 1e7: count 0.05, scan 0.02, scatter 0.12 ms, bound
// by random atomics and 4-byte stores in the L2, against 0.54 ms for the five
// 8-bit radix passes it replaced in the timestep (keys with the index packed
// into their low bits, histograms, tie fix).
// Stars crowding into few bins: a warp in which a thread finds all its four in one
// adds to each bin with its lanes together (atomics on one address go at 2.4 a
// nanosecond: 10^6 stars in two bins counted in 424 us, 28 so).  Two neighbours in
// one bin are common enough among few stars that the sort of 1021 would take 11.3
// us instead of 10.0.
__device__ __forceinline__ bool crowded(const uint4& b) {
  return __any_sync(__activemask(), b.x == b.y && b.y == b.z && b.z == b.w);
}
// this lane's place among the lanes that add to the same counter
__device__ __forceinline__ uint32_t add_together(uint32_t* a, uint32_t bin) {
  const unsigned peers = __match_any_sync(__activemask(), bin), lane = threadIdx.x & 31;
  const int first = __ffs(peers) - 1;
  uint32_t old = 0u;
  if ((int)lane == first) old = atomicAdd(a + bin, (uint32_t)__popc(peers));
  return __shfl_sync(peers, old, first) + __popc(peers & ((1u << lane) - 1u));
}

__global__ void __launch_bounds__(256) k_bin_count(int64_t n, const uint32_t* bin,
                                                   uint32_t* cnt) {
  pdl_enter();
  const int64_t p0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4;
  if (p0 + 4 <= n) {
    const uint4 b = *reinterpret_cast<const uint4*>(bin + p0);
    if (crowded(b)) {
      add_together(cnt, b.x);
      add_together(cnt, b.y);
      add_together(cnt, b.z);
      add_together(cnt, b.w);
      return;
    }
    atomicAdd(cnt + b.x, 1u);
    atomicAdd(cnt + b.y, 1u);
    atomicAdd(cnt + b.z, 1u);
    atomicAdd(cnt + b.w, 1u);
  } else {
    for (int64_t p = p0; p < n; ++p) atomicAdd(cnt + bin[p], 1u);
  }
}

// Exclusive scan of the counts in place, one pass: tiles of kBinTile bins in
// ticket order, the sum of the tiles before by decoupled look-back, one warp
// reading 32 tiles' words at a time.  Each wait is bounded (g_spin_cap polls
// of a window that is not complete).  Bins with more than kRunMax stars are
// listed, those with more than kRunTile with their share of the work's tiles.
__global__ void __launch_bounds__(kThreads) k_bin_scan(uint32_t* cnt, unsigned long long* desc,
                                                       uint32_t* ctl, uint2* runs, uint4* big,
                                                       uint32_t* err) {
  pdl_enter();
  __shared__ uint32_t s_warp[kWarps];
  __shared__ uint32_t s_tile, s_excl;
  constexpr int kPer = kBinTile / kThreads;  // 16 consecutive bins per thread
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) s_tile = atomicAdd(ctl + kCtlScan, 1u);
  __syncthreads();
  const int64_t t = s_tile;
  uint4* mine = reinterpret_cast<uint4*>(cnt + t * kBinTile + tid * kPer);
  uint4 c[kPer / 4];
  uint32_t sum = 0, most = 0;
#pragma unroll
  for (int i = 0; i < kPer / 4; ++i) {
    c[i] = mine[i];
    most = max(max(max(c[i].x, c[i].y), max(c[i].z, c[i].w)), most);
    sum += c[i].x + c[i].y + c[i].z + c[i].w;
  }
  const uint32_t before = block_excl_scan_u32(sum, s_warp);
  if (warp == 0) {
    const unsigned long long total = s_warp[kWarps - 1];
    uint32_t excl = 0;
    if (lane == 0) atomicExch(desc + t, (t == 0 ? kFlagInc : kFlagAgg) | total);
    const int cap = g_spin_cap;
    int spins = 0;
    int64_t j = t - 1;
    while (j >= 0) {
      const int64_t q = j - lane;
      const unsigned long long w = q >= 0 ? ld_volatile(desc + q) : kFlagInc;
      const unsigned ready = __ballot_sync(0xffffffffu, (w & ~kCountMask) != 0);
      const unsigned inc = __ballot_sync(0xffffffffu, (w & ~kCountMask) == kFlagInc);
      const unsigned use = inc ? (2u << (__ffs(inc) - 1)) - 1u : 0xffffffffu;
      if ((ready & use) != use) {
        if (++spins >= cap) {
          if (lane == 0) set_err(err, kErrTimeout);
          break;
        }
        if (spins > 32) __nanosleep(64);
        continue;
      }
      excl += __reduce_add_sync(0xffffffffu, (use >> lane) & 1u ? (uint32_t)(w & kCountMask) : 0u);
      if (inc) break;
      j -= 32;
    }
    if (lane == 0) {
      if (t) atomicExch(desc + t, kFlagInc | (excl + total));
      s_excl = excl;
    }
  }
  __syncthreads();
  uint32_t at = s_excl + before;
#pragma unroll
  for (int i = 0; i < kPer / 4; ++i) {
    uint32_t v[4] = {c[i].x, c[i].y, c[i].z, c[i].w}, o[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      o[k] = at;
      at += v[k];
    }
    mine[i] = make_uint4(o[0], o[1], o[2], o[3]);
  }
  if (most <= (uint32_t)kRunMax) return;
  const uint32_t* from = reinterpret_cast<const uint32_t*>(mine);
#pragma unroll 1
  for (int i = 0; i < kPer; ++i) {
    const uint32_t p = from[i], len = (i + 1 < kPer ? from[i + 1] : at) - p;
    if (len <= (uint32_t)kRunMax) continue;
    const uint32_t nt = (len + kRunTile - 1) / kRunTile;
    if (nt == 1u) {
      runs[atomicAdd(ctl + kCtlRuns, 1u)] = make_uint2(p, len);
    } else {
      atomicMax(ctl + kCtlMost, nt);
      const uint32_t b = atomicAdd(ctl + kCtlTiles, nt);
      big[atomicAdd(ctl + kCtlBig, 1u)] = make_uint4(p, len, b, b + nt);
    }
  }
}

// the stars' indices to their bins' positions (the order inside a bin is
// whatever the atomics give; the gather settles it)
__global__ void __launch_bounds__(256) k_bin_scatter(int64_t n, const uint32_t* bin,
                                                     uint32_t* at, uint32_t* order,
                                                     uint32_t* err) {
  pdl_enter();
  const int64_t p0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4;
  auto put = [&](uint32_t pos, int64_t p) {
    if ((int64_t)pos < n) order[pos] = (uint32_t)p;
    else set_err(err, kErrTimeout);  // only after a timed-out look-back
  };
  if (p0 + 4 <= n) {
    const uint4 b = *reinterpret_cast<const uint4*>(bin + p0);
    uint32_t a0, a1, a2, a3;
    if (crowded(b)) {
      a0 = add_together(at, b.x), a1 = add_together(at, b.y);
      a2 = add_together(at, b.z), a3 = add_together(at, b.w);
    } else {
      a0 = atomicAdd(at + b.x, 1u), a1 = atomicAdd(at + b.y, 1u);
      a2 = atomicAdd(at + b.z, 1u), a3 = atomicAdd(at + b.w, 1u);
    }
    put(a0, p0);
    put(a1, p0 + 1);
    put(a2, p0 + 2);
    put(a3, p0 + 3);
  } else {
    for (int64_t p = p0; p < n; ++p) put(atomicAdd(at + bin[p], 1u), p);
  }
}

// The listed runs (more than kRunMax stars in one bin: new radii crowding
// into one shell of the old table, as when a thin shell of stars spreads out)
// in (r, id) order.  A step without such runs finds the lists empty.
//
// A run of up to kRunTile stars is sorted by one block in shared memory.  A longer
// one is a merge sort over all blocks: its tiles are sorted like that, then every
// pass merges pairs of sorted stretches, one tile of the result per block, whose
// part of the two stretches a search along the merge's diagonal finds.  (r, id) is
// a strict order, so the result is the one order whatever the input's, which the
// scatter's atomics decide.  Blocks take their work by ticket in the order tiles,
// short runs, first pass, second pass ...; a tile of a pass waits until all of the
// pass before it are done, which were all taken by blocks that run already.
// Each wait is bounded (g_spin_cap polls).
//
// Nearly all stars in two runs, sort stage of 3 x 10^4, 2 x 10^5, 10^6, 10^7 stars: 0.10,
// 0.16, 0.30, 2.3 ms (at 10^6 0.24 of it this kernel); by the radix passes 0.07, 0.08,
// 0.13, 0.76; with one block to a run, as the first three were before, 0.76, 5.2, 27.
constexpr int64_t kRunBlocks = 608;  // four to an SM (two: the million's 0.28 ms)
struct RunSmem {
  unsigned long long key[kRunTile];
  uint32_t idx[kRunTile], id[kRunTile];
  uint32_t item, cut[2];
  uint4 run;
  bool ok;
};

// order[0 .. len) -> out, by (r, id); keys (may be null): the bits of r
__device__ __forceinline__ void sort_run_tile(RunSmem& S, const RecA* rec, const uint32_t* in,
                                              uint32_t* out, unsigned long long* keys,
                                              uint32_t len) {
  const uint32_t tid = threadIdx.x;
  uint32_t size = 64;
  while (size < len) size <<= 1;
  for (uint32_t i = tid; i < size; i += kThreads) {
    const uint32_t v = i < len ? in[i] : 0u;
    if (i < len) {
      const RecA A = load_rec(rec + v);
      S.key[i] = ubits(A.r);
      S.id[i] = A.id;
    } else {
      S.key[i] = ~0ull;  // (above every radius: stays at the end)
      S.id[i] = ~0u;
    }
    S.idx[i] = v;
  }
  __syncthreads();
  // bitonic sort; a warp's 32 pairs lie in 64 neighbours while j <= 32
  for (uint32_t k = 2; k <= size; k <<= 1)
    for (uint32_t j = k >> 1; j > 0; j >>= 1) {
      for (uint32_t t = tid; t < size / 2; t += kThreads) {
        const uint32_t a = 2 * t - (t & (j - 1)), b = a + j;
        const unsigned long long ka = S.key[a], kb = S.key[b];
        const uint32_t ia = S.id[a], ib = S.id[b];
        const bool a_first = ka < kb || (ka == kb && ia < ib);
        if (a_first != ((a & k) == 0u)) {
          S.key[a] = kb;
          S.key[b] = ka;
          S.id[a] = ib;
          S.id[b] = ia;
          const uint32_t v = S.idx[a];
          S.idx[a] = S.idx[b];
          S.idx[b] = v;
        }
      }
      if (j > 32 || (j == 1 && k >= 64)) __syncthreads();
      else __syncwarp();
    }
  for (uint32_t i = tid; i < len; i += kThreads) {
    out[i] = S.idx[i];
    if (keys) keys[i] = S.key[i];
  }
}

struct RunBuf {
  unsigned long long* key;
  uint32_t* idx;
};

// Of the first d of the merge of stretches a (na) and b (nb), how many come from
// a: by one warp, 32 probes a round.  (Written by other blocks of this kernel: read
// past the L1.)
__device__ __forceinline__ uint32_t merge_cut(const RunBuf& in, const RecA* rec, uint32_t a,
                                              uint32_t na, uint32_t b, uint32_t nb, uint32_t d) {
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t lo = d > nb ? d - nb : 0u, hi = d < na ? d : na;
  while (lo < hi) {
    const unsigned long long span = hi - lo;
    const uint32_t m = lo + (uint32_t)(span * lane / 32u);
    const uint32_t pa = a + m, pb = b + (d - 1u - m);
    const unsigned long long ka = __ldcg(in.key + pa), kb = __ldcg(in.key + pb);
    const bool from_a =
        ka < kb || (ka == kb && rec[__ldcg(in.idx + pa)].id < rec[__ldcg(in.idx + pb)].id);
    const uint32_t k = (uint32_t)__popc(__ballot_sync(0xffffffffu, from_a));
    // the first k probes come from a (probes rise with the lane)
    if (k == 0) return lo;
    hi = k == 32u ? hi : lo + (uint32_t)(span * k / 32u);
    lo = lo + (uint32_t)(span * (k - 1u) / 32u) + 1u;
  }
  return lo;
}

// tile t of a run of len stars from first on: merged from the stretches of width w
__device__ __forceinline__ void merge_run_tile(RunSmem& S, const RecA* rec, const RunBuf& in,
                                               const RunBuf& out, uint32_t first, uint32_t len,
                                               uint32_t t, uint32_t w) {
  const uint32_t tid = threadIdx.x, o = t * kRunTile, pair = o / (2u * w) * (2u * w);
  const uint32_t rest = len - pair;  // (w <= len: the last pass has 2 w >= len > w)
  const uint32_t na = rest < w ? rest : w, nb = rest - na < w ? rest - na : w;
  const uint32_t a = first + pair, b = a + na;
  const uint32_t d0 = o - pair;
  const uint32_t d1 = d0 + kRunTile < na + nb ? d0 + kRunTile : na + nb;
  if (tid < 64) {
    const uint32_t cut = merge_cut(in, rec, a, na, b, nb, tid < 32 ? d0 : d1);
    if ((tid & 31u) == 0u) S.cut[tid >> 5] = cut;
  }
  __syncthreads();
  const uint32_t c0 = S.cut[0], ta = S.cut[1] - c0, all = d1 - d0, tb = all - ta;
  for (uint32_t i = tid; i < all; i += kThreads) {
    const uint32_t p = i < ta ? a + c0 + i : b + (d0 - c0) + (i - ta);
    S.key[i] = __ldcg(in.key + p);
    S.idx[i] = __ldcg(in.idx + p);
  }
  __syncthreads();
  auto from_a = [&](uint32_t x, uint32_t y) {
    const unsigned long long ka = S.key[x], kb = S.key[y];
    return ka < kb || (ka == kb && rec[S.idx[x]].id < rec[S.idx[y]].id);
  };
  constexpr uint32_t kPer = kRunTile / kThreads;
  const uint32_t e = tid * kPer;
  unsigned long long k[kPer];
  uint32_t v[kPer];
  if (e < all) {
    uint32_t lo = e > tb ? e - tb : 0u, hi = e < ta ? e : ta;
    while (lo < hi) {
      const uint32_t m = (lo + hi) >> 1;
      if (from_a(m, ta + (e - 1u - m))) lo = m + 1u; else hi = m;
    }
    uint32_t x = lo, y = ta + (e - lo);
#pragma unroll
    for (uint32_t i = 0; i < kPer; ++i) {
      const bool left = x < ta && (y >= all || from_a(x, y));
      const uint32_t q = left ? x++ : (y < all ? y++ : all - 1u);  // (past the end: not stored)
      k[i] = S.key[q];
      v[i] = S.idx[q];
    }
  }
  __syncthreads();
  if (e < all) {
#pragma unroll
    for (uint32_t i = 0; i < kPer; ++i) {
      S.key[e + i] = k[i];
      S.idx[e + i] = v[i];
    }
  }
  __syncthreads();
  for (uint32_t i = tid; i < all; i += kThreads) {
    out.key[first + o + i] = S.key[i];
    out.idx[first + o + i] = S.idx[i];
  }
}

// the listed runs' work, by all blocks; false: a wait gave up
__device__ __forceinline__ bool long_runs(RunSmem& S, uint32_t* ctl, const uint2* runs,
                                          const uint4* big, const RecA* rec, const RunBuf& home,
                                          const RunBuf& away, uint32_t nr, uint32_t nt,
                                          uint32_t* err) {
  const uint32_t passes = nt ? 32u - (uint32_t)__clz((int)(ctl[kCtlMost] - 1u)) : 0u;
  const uint32_t total = nt + nr + passes * nt, nb = ctl[kCtlBig];
  const int cap = g_spin_cap;
  // the long run that tile i belongs to: first star, length, tile there
  auto run_of = [&](uint32_t i) {
    for (uint32_t l = threadIdx.x; l < nb; l += kThreads) {
      const uint4 t = big[l];
      if (t.z <= i && i < t.w) S.run = make_uint4(t.x, t.y, i - t.z, 0u);
    }
    __syncthreads();
    return S.run;
  };
  for (;;) {
    if (threadIdx.x == 0) S.item = atomicAdd(ctl + kCtlNext, 1u);
    __syncthreads();
    const uint32_t item = S.item;
    if (item >= total) return true;
    if (item >= nt && item < nt + nr) {
      const uint2 run = runs[item - nt];
      sort_run_tile(S, rec, home.idx + run.x, home.idx + run.x, nullptr, run.y);
      __syncthreads();
      continue;
    }
    if (item < nt) {
      // the passes end at home
      const RunBuf& out = passes & 1u ? away : home;
      const uint4 t = run_of(item);
      const uint32_t o = t.z * kRunTile, len = t.y - o < kRunTile ? t.y - o : kRunTile;
      sort_run_tile(S, rec, home.idx + t.x + o, out.idx + t.x + o, out.key + t.x + o, len);
    } else {
      const uint32_t q = (item - nt - nr) / nt;
      if (threadIdx.x == 0) {
        int spins = 0;
        S.ok = true;
        while (*(volatile uint32_t*)(ctl + kCtlDone) < (q + 1u) * nt) {
          if (++spins > cap || (*(volatile uint32_t*)err & kErrTimeout)) {
            set_err(err, kErrTimeout);
            S.ok = false;
            break;
          }
          if (spins > 32) __nanosleep(64);
        }
        __threadfence();
      }
      __syncthreads();
      if (!S.ok) return false;
      const uint4 t = run_of((item - nt - nr) % nt);
      const bool from_home = ((passes ^ q) & 1u) == 0u;
      merge_run_tile(S, rec, from_home ? home : away, from_home ? away : home, t.x, t.y, t.z,
                     (uint32_t)kRunTile << q);
    }
    __threadfence();  // this tile before its mark
    __syncthreads();
    if (threadIdx.x == 0) atomicAdd(ctl + kCtlDone, 1u);
  }
}

__global__ void __launch_bounds__(kThreads) k_long_runs(int64_t n, uint32_t* ctl,
                                                        const uint2* runs, const uint4* big,
                                                        const RecA* rec, RunBuf home, RunBuf away,
                                                        uint32_t* err) {
  pdl_enter();
  const uint32_t nr = ctl[kCtlRuns], nt = ctl[kCtlTiles];
  bool lost = *err & kErrTimeout;
  if (nr + nt == 0u && !lost) return;
  __shared__ RunSmem S;
  if (!lost) long_runs(S, ctl, runs, big, rec, home, away, nr, nt, err);
  // After a wait that gave up, here or in the scan, the order is not a permutation:
  // the last block to leave puts the stars where they are, so that what follows up
  // to the report reads stars only.
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    S.ok = atomicAdd(ctl + kCtlLeft, 1u) == gridDim.x - 1u &&
           (*(volatile uint32_t*)err & kErrTimeout);
    __threadfence();
  }
  __syncthreads();
  if (S.ok)
    for (int64_t p = threadIdx.x; p < n; p += kThreads) home.idx[p] = (uint32_t)p;
}

__global__ void k_philox(int64_t n, const uint32_t* ctr, uint64_t seed, uint32_t* out) {
  pdl_enter();
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint4 c = reinterpret_cast<const uint4*>(ctr)[i];
  U4 w = philox(c.x, c.y, c.z, c.w, seed);
  reinterpret_cast<uint4*>(out)[i] = make_uint4(w.x, w.y, w.z, w.w);
}

template <bool kId, int IPT, int kRank>
void set_pass_smem() {
  cudaFuncSetAttribute(k_pass<kId, IPT, kRank>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)sizeof(PassSmem<IPT>));
}

template <int IPT, int kRank>
void launch_pass(const SegLayout& L, SortWork& W, bool id, const uint64_t* kin,
                 const uint32_t* vin, uint64_t* kout, uint32_t* vout, int pass, int q,
                 int passes, uint32_t* err, cudaStream_t st) {
  const unsigned grid = (unsigned)W.n_stiles;
  const size_t sm = sizeof(PassSmem<IPT>);
  launch_k(id ? k_pass<true, IPT, kRank> : k_pass<false, IPT, kRank>, grid, kThreads, sm, st,
           L.off, W.stile_off, L.n_seg, W.n_stiles, kin, vin, kout, vout, pass, q, passes,
           W.hist, W.desc, W.tickets, err);
}

}  // namespace

// ------------------------------------------------------------------ host
cudaError_t set_wait_limits(int spin_polls, long long tie_moves) {
  const int sp = spin_polls > 0 ? spin_polls : kSpinCapDefault;
  const long long tm = tie_moves > 0 ? tie_moves : kTieMoveCapDefault;
  cudaError_t e = cudaMemcpyToSymbol(g_spin_cap, &sp, sizeof(sp));
  if (!e) e = cudaMemcpyToSymbol(g_tie_move_cap, &tm, sizeof(tm));
  return e;
}

void sort_prepare() {
  set_pass_smem<true, 8, kRankMatch>();
  set_pass_smem<false, 8, kRankMatch>();
  set_pass_smem<true, 8, kRankBallot>();
  set_pass_smem<false, 8, kRankBallot>();
  set_pass_smem<true, 16, kRankMatch>();
  set_pass_smem<false, 16, kRankMatch>();
  set_pass_smem<true, 16, kRankBallot>();
  set_pass_smem<false, 16, kRankBallot>();
  cudaFuncSetAttribute(k_upsweep, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)(sizeof(uint32_t) * kWarps * kMaxPasses * kBins));
}

static std::vector<int64_t> sort_tile_offsets(const SegLayout& L, int tile) {
  std::vector<int64_t> o(L.n_seg + 1, 0);
  for (int c = 0; c < L.n_seg; ++c) {
    const int64_t nc = L.h_off[c + 1] - L.h_off[c];
    o[c + 1] = o[c] + (nc + tile - 1) / tile;
  }
  return o;
}

cudaError_t sort_set_shape(const SegLayout& L, SortWork& W, int ipt, int rank,
                           cudaStream_t st) {
  if ((ipt != 8 && ipt != 16) || (rank != 0 && rank != 1))
    return cudaErrorInvalidValue;
  std::vector<int64_t> o = sort_tile_offsets(L, kThreads * ipt);
  cudaError_t e = cudaMemcpyAsync(W.stile_off, o.data(), sizeof(int64_t) * o.size(),
                                  cudaMemcpyHostToDevice, st);
  if (!e) e = cudaStreamSynchronize(st);  // o lives on this stack
  if (e) return e;
  W.ipt = ipt;
  W.rank = rank;
  W.n_stiles = o[L.n_seg];
  return cudaSuccess;
}

// Histograms, tickets and done counters first, then the look-back words: a sort
// zeroes the counters and the words of its own passes and tiles.
static size_t sort_head_bytes(const SegLayout& L, int max_passes) {
  const size_t hist = sizeof(uint32_t) * (size_t)L.n_seg * max_passes * kBins;
  return (hist + sizeof(uint32_t) * (16 + (size_t)L.n_seg) + 255) / 256 * 256;
}
size_t sort_zeroed_bytes(const SegLayout& L, int max_passes) {
  // look-back words for the smallest tiles (the most tiles)
  const int64_t max_tiles = sort_tile_offsets(L, kThreads * 8)[L.n_seg];
  return sort_head_bytes(L, max_passes) +
         sizeof(unsigned long long) * (size_t)max_passes * max_tiles * kBins;
}

cudaError_t alloc_sort(SortWork& W, const SegLayout& L, int max_passes, cudaStream_t st,
                       uint64_t* keys, void* zeroed) {
  W.max_passes = max_passes;
  W.zero_head = sort_head_bytes(L, max_passes);
  W.ipt = 16;
  W.rank = 0;
  const std::vector<int64_t> o = sort_tile_offsets(L, kThreads * W.ipt);
  W.n_stiles = o[L.n_seg];
  unsigned char* own = nullptr;
  Carve C;
  C.put(W.stile_off, o.data(), o.size());
  C.add(W.vals_alt, (size_t)L.n);
  if (!keys) C.add(W.keys_alt, (size_t)L.n);
  if (!zeroed) C.add(own, sort_zeroed_bytes(L, max_passes));
  const cudaError_t e = C.alloc(W.block, st);
  if (e) return e;
  if (keys) W.keys_alt = keys;
  unsigned char* base = zeroed ? (unsigned char*)zeroed : own;
  W.zero_base = base;
  W.hist = (uint32_t*)base;
  W.tickets = W.hist + (size_t)L.n_seg * max_passes * kBins;
  W.done = W.tickets + 16;
  W.desc = (unsigned long long*)(base + W.zero_head);
  return cudaSuccess;
}

void free_sort(SortWork& W, cudaStream_t st) {
  if (W.block) cudaFreeAsync(W.block, st);
  W = SortWork();
}

cudaError_t sort_segments(const SegLayout& L, SortWork& W, uint64_t* keys, uint32_t* vals,
                          int first_pass, int passes, bool vals_identity, uint32_t* err,
                          cudaStream_t st, uint64_t** keys_res, uint32_t** vals_res) {
  if (keys_res) *keys_res = keys;
  if (vals_res) *vals_res = vals;
  if (passes <= 0 || passes > W.max_passes || L.n_tiles == 0) return cudaSuccess;
  cudaMemsetAsync(W.zero_base, 0,
                  W.zero_head + sizeof(unsigned long long) * (size_t)passes *
                                    (size_t)W.n_stiles * kBins,
                  st);
  launch_k(k_upsweep, (unsigned)L.n_tiles, kThreads, sizeof(uint32_t) * kWarps * passes * kBins, st,
      L.off, L.tile_off, L.n_seg, keys, first_pass, passes, W.hist, W.done);
  uint64_t* kin = keys;
  uint32_t* vin = vals;
  uint64_t* kout = W.keys_alt;
  uint32_t* vout = W.vals_alt;
  for (int q = 0; q < passes; ++q) {
    const bool id = q == 0 && vals_identity;
    const int pass = first_pass + q;
    if (W.ipt == 8 && W.rank == kRankMatch)
      launch_pass<8, kRankMatch>(L, W, id, kin, vin, kout, vout, pass, q, passes, err, st);
    else if (W.ipt == 8)
      launch_pass<8, kRankBallot>(L, W, id, kin, vin, kout, vout, pass, q, passes, err, st);
    else if (W.rank == kRankMatch)
      launch_pass<16, kRankMatch>(L, W, id, kin, vin, kout, vout, pass, q, passes, err, st);
    else
      launch_pass<16, kRankBallot>(L, W, id, kin, vin, kout, vout, pass, q, passes, err, st);
    std::swap(kin, kout);
    std::swap(vin, vout);
  }
  // after an odd number of passes the result is in the alternate buffers:
  // the caller takes them, or they are copied back
  if (kin != keys) {
    if (keys_res && vals_res) {
      *keys_res = kin;
      *vals_res = vin;
    } else {
      cudaMemcpyAsync(keys, kin, sizeof(uint64_t) * (size_t)L.n, cudaMemcpyDeviceToDevice, st);
      cudaMemcpyAsync(vals, vin, sizeof(uint32_t) * (size_t)L.n, cudaMemcpyDeviceToDevice,
                        st);
    }
  }
  return cudaPeekAtLastError();  // (left for the caller's own look)
}

void launch_tiefix(const SegLayout& L, uint64_t* keys, uint32_t* vals,
                   const uint32_t* ids_by_val, int id_stride, uint32_t* err,
                   cudaStream_t st, int shift) {
  if (L.n == 0) return;
  launch_k(k_tiefix, (unsigned)((L.n + 255) / 256), 256, 0, st,
      L.off, L.n_seg, L.n, keys, vals, ids_by_val, id_stride, shift, err, L.stats);
}

cudaError_t alloc_bins(BinWork& B, const SegLayout& L, cudaStream_t st) {
  std::vector<int64_t>& o = B.h_cbase;
  o.assign(L.n_seg + 1, 0);
  for (int c = 0; c < L.n_seg; ++c) {
    const int64_t nc = L.h_off[c + 1] - L.h_off[c];
    o[c + 1] = o[c] + (nc + 1) + (nc / 8 + 1);  // shells -1 .. nc - 1, then escapers by id
  }
  B.n_tiles = (o[L.n_seg] + kBinTile - 1) / kBinTile;
  B.n_bins = B.n_tiles * kBinTile;
  cudaError_t e;
  if ((e = cudaMallocAsync((void**)&B.cbase, sizeof(int64_t) * o.size(), st))) return e;
  if ((e = cudaMallocAsync((void**)&B.esh, sizeof(int) * L.n_seg, st))) return e;
  if ((e = cudaMallocAsync((void**)&B.cnt, sizeof(uint32_t) * B.n_bins, st))) return e;
  if ((e = cudaMallocAsync((void**)&B.desc, sizeof(unsigned long long) * B.n_tiles, st))) return e;
  if ((e = cudaMallocAsync((void**)&B.ctl, sizeof(uint32_t) * kCtlWords, st))) return e;
  if ((e = cudaMallocAsync((void**)&B.runs, sizeof(uint2) * (L.n / kRunMax + 1), st))) return e;
  if ((e = cudaMallocAsync((void**)&B.big, sizeof(uint4) * (L.n / kRunTile + 1), st)))
    return e;
  e = cudaMemcpyAsync(B.cbase, o.data(), sizeof(int64_t) * o.size(), cudaMemcpyHostToDevice, st);
  if (!e) e = cudaMemsetAsync(B.cnt, 0, sizeof(uint32_t) * B.n_bins, st);
  if (!e) e = cudaMemsetAsync(B.desc, 0, sizeof(unsigned long long) * B.n_tiles, st);
  if (!e) e = cudaMemsetAsync(B.ctl, 0, sizeof(uint32_t) * kCtlWords, st);
  if (e) return e;
  const std::vector<unsigned int> any((size_t)L.n_seg, 0xFFFFFFFFu);
  return set_bin_ids(B, L, any.data(), st);
}

void free_bins(BinWork& B, cudaStream_t st) {
  void* ps[] = {B.cbase, B.esh, B.cnt, B.desc, B.ctl, B.runs, B.big};
  for (void* p : ps)
    if (p) cudaFreeAsync(p, st);
  B = BinWork();
}

cudaError_t set_bin_ids(BinWork& B, const SegLayout& L, const unsigned int* max_id,
                        cudaStream_t st) {
  std::vector<int> sh((size_t)L.n_seg, 0);
  for (int c = 0; c < L.n_seg; ++c) {
    const int64_t nc = L.h_off[c + 1] - L.h_off[c];
    while (((uint64_t)max_id[c] >> sh[c]) > (uint64_t)(nc / 8)) ++sh[c];
  }
  cudaError_t e = cudaMemcpyAsync(B.esh, sh.data(), sizeof(int) * sh.size(),
                                  cudaMemcpyHostToDevice, st);
  if (!e) e = cudaStreamSynchronize(st);  // sh lives on this stack
  return e;
}

void launch_bin_sort(const SegLayout& L, BinWork& B, const uint32_t* bin, const RecA* rec,
                     uint32_t* order, uint32_t* scratch, uint64_t* keys, uint64_t* keys_scratch,
                     bool counted, uint32_t* err, cudaStream_t st) {
  if (L.n == 0) return;
  const unsigned grid = (unsigned)((L.n + 1023) / 1024);
  if (!counted) launch_k(k_bin_count, grid, 256, 0, st, L.n, bin, B.cnt);
  launch_k(k_bin_scan, (unsigned)B.n_tiles, kThreads, 0, st, B.cnt, B.desc, B.ctl, B.runs, B.big,
           err);
  launch_k(k_bin_scatter, grid, 256, 0, st, L.n, bin, B.cnt, order, err);
  const int64_t most = L.n / kRunMax + 1;  // listed runs at most
  const RunBuf home{reinterpret_cast<unsigned long long*>(keys), order};
  const RunBuf away{reinterpret_cast<unsigned long long*>(keys_scratch), scratch};
  launch_k(k_long_runs, (unsigned)(most < kRunBlocks ? most : kRunBlocks), kThreads, 0, st, L.n,
           B.ctl, B.runs, B.big, rec, home, away, err);
}

void launch_philox(int64_t n, const uint32_t* ctr, uint64_t seed, uint32_t* out,
                   cudaStream_t st) {
  if (n <= 0) return;
  launch_k(k_philox, (unsigned)((n + 255) / 256), 256, 0, st, n, ctr, seed, out);
}

CMC_DEBUG_SITE_ACCESSOR

}  // namespace cmc
