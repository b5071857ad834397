// Values of the potential grid and the slopes at the tile seams: a part of the
// tables that k_grid_build (stage calls, set states) and, beside its own work,
// k_phi_old (timesteps) write.
#pragma once
#include "cmc_host.hpp"

namespace cmc {

__device__ __forceinline__ double2 node_xp(const double4_32a* p) {
  return *reinterpret_cast<const double2*>(p);
}

// Phi at every grid key from the FP64 table: Phi = Phi_i + M_i (1/r_i - 1/r)
// in the key's shell i (Eq. 6 with the enclosed-mass slope), Phi_0 inside
// the first star, rounded to float
// fused (launch_potential_tables): the slopes at the tile seams, which the
// potential kernel leaves, are computed here by n_tiles more threads (and
// locally where a cell needs one), and each segment's cell 0 fills Phi_0 and
// the bound mass into gaux
// p: a cell or, from `total` on, a tile (whole warps call it).
__device__ __forceinline__ void grid_build(const Seg& S, const int64_t* esc, const GridBuild& A,
                                           int64_t p) {
  const double* x = A.x;
  const double* phi = A.phi;
  const BucketArgs& B = A.B;
  const int* gshell = A.gshell;
  float* gphi = A.gphi;
  float4* gaux = A.gaux;
  const int64_t total = A.total, n_tiles = A.n_tiles;
  const bool fused = A.fused, sub = A.sub;
  double4_32a* node = A.node;
  const unsigned am = __ballot_sync(0xFFFFFFFFu, p < total);
  if (p >= total) {
    const int64_t t = p - total;
    if (!fused || t >= n_tiles) return;
    const int cs = seg_find(S.tile_off, S.n_seg, t);
    const int64_t sbs = S.off[cs], nbs = S.nb[cs] - (sub ? esc[cs] : 0);
    const int64_t k = (t - S.tile_off[cs]) * kTile + kTile - 1;  // the tile's last star
    if (k + 1 >= nbs) return;
    const int64_t q = sbs + k;
    // (only the slope: other threads read the record's 1/r and Phi)
    node[q].w = div_rn(phi[q + 1] - phi[q], x[q] - x[q + 1]);
    return;
  }
  const int c = seg_find(B.goff, S.n_seg, p);
  const int4 pr = B.gprm[c];
  const int g = (int)(p - B.goff[c]);
  const int64_t sb = S.off[c];
  const int64_t nb = S.nb[c] - (sub ? esc[c] : 0);
  // shell i's slope (a seam's computed as the seam threads do)
  auto slope = [&](int64_t i) {
    if (fused && i % kTile == kTile - 1 && i + 1 < nb) {
      const double2 a = node_xp(node + sb + i), b = node_xp(node + sb + i + 1);
      return div_rn(b.y - a.y, a.x - b.x);
    }
    return node[sb + i].w;
  };
  float rel = 0.0f;
  if (g < pr.z) {
    if (fused && g == 0) {
      gaux[c].x = (float)phi[sb];
      gaux[c].y = (float)node[sb + nb - 1].w;
    }
    const double xg = (double)__uint_as_float((uint32_t)pr.x + ((uint32_t)g << pr.y));
    const double xn = (double)__uint_as_float((uint32_t)pr.x + ((uint32_t)(g + 1) << pr.y));
    const int64_t lo = gshell[p];
    double ph = phi[sb];
    if (lo >= 0) {
      const double2 a = node_xp(node + sb + lo);
      ph = a.y + slope(lo) * (a.x - xg);
    }
    gphi[p] = (float)ph;
    // Phi is convex in 1/r (its slope -M(1/r) rises with 1/r), so inside the
    // cell [xg, xn] it lies below the chord by at most (xn - xg) dM / 4, dM
    // the mass of the stars in the cell; relative to |Phi(xg)|, the smallest
    // |Phi| of the cell, the largest over the segment's cells bounds the
    // grid's interpolation error (gaux.w; floats >= 0 order as their bits)
    if (g + 1 < pr.z && ph < 0.0) {
      const int64_t lo2 = gshell[p + 1];
      const double Ma = lo < 0 ? 0.0 : slope(lo);
      const double Mb = lo2 < 0 ? 0.0 : slope(lo2);
      const double dM = Ma - Mb;
      rel = (float)(((xn - xg) * (dM > 0.0 ? dM : 0.0) * 0.25) / -ph);
    }
  }
  // one atomic per segment present in the warp
  const unsigned grp = __match_any_sync(am, c);
  const unsigned mx = __reduce_max_sync(grp, __float_as_uint(rel));
  if ((threadIdx.x & 31) == (unsigned)(__ffs(grp) - 1) && mx)
    atomicMax(reinterpret_cast<unsigned int*>(&gaux[c].w), mx);
}

}  // namespace cmc
