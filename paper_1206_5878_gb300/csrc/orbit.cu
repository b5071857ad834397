// New orbits (section 2.1 step 5, Eqs. 12-15; Appendix A's bisection and
// rejection kernels, fused): one thread per star.
//
//   E = Phi_k + (v_r^2 + v_t^2)/2,  J = r_k v_t;  E >= 0: the star escapes.
//   r_max, r_min: bisection over the star nodes for the sign change of
//   Q(r) = 2E - 2 Phi(r) - J^2/r^2 (Eq. 12), then the root of Q inside the
//   shell, where Eq. 6 makes Phi = A - B/r.
//   New radius: von Neumann rejection (Eqs. 14-15) in the variable s of
//   r(s) = (rmax+rmin)/2 + (rmax-rmin)/4 (3s - s^3), whose density
//   g(s) = (dr/ds)/sqrt(Q) stays finite at both turning points; the bound
//   is F = 1.2 max_j g(s_j) on s_j = -1 + (j + 1/2)/10.5, j = 0..20.
//   v_t = J/r_new, v_r = +-sqrt(Q(r_new)).
//
// precision 0 (FP64): every result is that of the FP64 operations of the
// method's statement, in the same order (searches and accept tests screened in
// floats with error bounds), so it is bit-identical to it.  precision 1
// (mixed): the same turning points; the bound F and the accept tests run in
// FP32 on the potential grid, the trials they cannot decide in FP64, and the
// accepted radius, its potential (by the shell's slope) and the velocities are
// FP64.  A mixed result matches the FP64 result to rounding whenever both
// accept the same trial.
#include "grid_build.cuh"

namespace cmc {

namespace {

struct Star {
  double E, J;
  int64_t k;
};

__device__ __forceinline__ double Q_node64(const Table64& T, const Star& s, int64_t i) {
  double L = s.J * T.x[i];
  return scale_up<1>(s.E - T.phi[i]) - L * L;
}

// root of Q inside shell j (nodes j, j+1; node nb is 1/r = 0, Phi = 0)
__device__ __forceinline__ double shell_root64(const Table64& T, const Star& s, int64_t j,
                                               bool outer) {
  const double rj = T.r[j], xj = T.x[j], pj = T.phi[j];
  double rj1, xj1, pj1;
  const bool has_next = j + 1 < T.nb;
  if (has_next) { rj1 = T.r[j + 1]; xj1 = T.x[j + 1]; pj1 = T.phi[j + 1]; }
  else { rj1 = __longlong_as_double(0x7FF0000000000000ll); xj1 = 0.0; pj1 = 0.0; }
  if (!(xj - xj1 > 0.0)) return rj;
  const double B = div_rn(pj1 - pj, xj - xj1);
  const double A = pj + B * xj;
  double D = B * B + scale_up<1>(s.J * s.J) * (s.E - A);
  if (!(D > 0.0)) D = 0.0;
  const double sD = sqrt_rn(D);
  double root = outer ? div_rn(B + sD, scale_up<1>(A - s.E)) : div_rn(s.J * s.J, B + sD);
  if (!(root >= rj)) root = rj;
  if (has_next && root > rj1) root = rj1;
  return root;
}

// The same root with the slope of shell j taken from the enclosed mass:
// across shell j, (Phi_{j+1} - Phi_j)/(x_j - x_{j+1}) = G M_j exactly
// (Eqs. 1-5; for the outermost shell M_j is the bound mass), so
// Phi = Phi_j + M_j (x_j - x) needs no division (mixed mode).  The cores
// take the node values, so that values loaded ahead and the table give
// the same arithmetic.  The clamps are the FP64 comparisons restated on
// the bit patterns (radii are positive).  Their quotients and square roots
// run on the integer pipes: this kernel is bound by the FP64 pipe first
// (turning points 1.30 ms with the square roots on the FP64 pipe, 1.275 ms
// without, at N = 10^7; 0.127 and 0.111 ms at 10^6, where the tables stay in
// the L2).
__device__ __forceinline__ double rmax_core(const Star& s, double rj, double xj, double pj,
                                            double Mj, bool has_next, double rj1) {
  const double B = Mj;
  const double A = pj + B * xj;
  const double em = s.E - A;
  double D = B * B + scale_up<1>(s.J * s.J) * em;
  if (!pos_num(D)) D = 0.0;
  const double sD = sqrt_rn(D);
  // 2 (A - E) = -(2 (E - A)) exactly
  double root = div_rn(B + sD, -scale_up<1>(em));
  if (!ge_pos(root, rj)) root = rj;
  if (has_next && ubits(root) > ubits(rj1)) root = rj1;
  return root;
}

// r_min in mixed mode: the shell root, or inside the innermost node
// (central, where Phi = Phi_0) J / sqrt(2 (E - Phi_0)) as central_root64
// computes it; both take one square root and one division, so the two
// cases share them (B = 0 makes B + sqrt(D) the bare root) and a warp
// holding both kinds of star runs them once.  Central: node values of
// node 0 and rj = r_0.
__device__ __forceinline__ double rmin_core(const Star& s, bool central, double rj, double xj,
                                            double pj, double Mj, bool has_next, double rj1) {
  const double B = central ? 0.0 : Mj;
  double D, num;
  if (central) {
    D = scale_up<1>(s.E - pj);
    num = s.J;
  } else {
    const double A = pj + B * xj;
    D = B * B + scale_up<1>(s.J * s.J) * (s.E - A);
    if (!pos_num(D)) D = 0.0;
    num = s.J * s.J;
  }
  double root = div_rn(num, B + sqrt_rn(D));
  if (central) {
    // root >= 0 (-0 included, NaN not), then root <= r_0
    const unsigned long long u = ubits(root);
    if (!(u <= kInfBits || u == 0x8000000000000000ull)) root = 0.0;
    if (__double_as_longlong(root) > __double_as_longlong(rj)) root = rj;
  } else {
    if (!ge_pos(root, rj)) root = rj;
    if (has_next && ubits(root) > ubits(rj1)) root = rj1;
  }
  return root;
}

// The FP64 shell of q (largest i with r_i <= q, -1 if none; integer
// compares of the radii's bits) from a guess i by a bounded walk, then a
// bisection, on the node records; a receives that shell's record (node 0's
// for -1).  The records of the guess and its successor are loaded together.
__device__ __forceinline__ int64_t fix_shell_nodes(const double4_32a* nd, int64_t nb,
                                                   int64_t i, double q, double4_32a& a) {
  if (!ge0(q)) {
    a = nd[0];
    return -1;
  }
  if (i < -1) i = -1;
  if (i >= nb) i = nb - 1;
  const long long qb = dbits(q);
  if (!CMC_IN(i < 0 ? 0 : i, nb)) i = -1;
  a = nd[i < 0 ? 0 : i];
  double4_32a b = i + 1 < nb ? nd[i + 1] : a;
  for (int w = 0; w < 64; ++w) {
    if (i + 1 < nb && dbits(b.z) <= qb) {
      ++i;
      a = b;
      if (i + 1 < nb) b = nd[i + 1];
      continue;
    }
    if (i >= 0 && dbits(a.z) > qb) {
      --i;
      b = a;
      a = nd[i < 0 ? 0 : i];
      continue;
    }
    return i;
  }
  int64_t lo = -1, hi = nb;
  while (hi - lo > 1) {
    const int64_t mid = lo + ((hi - lo) >> 1);
    if (dbits(nd[mid].z) <= qb) lo = mid; else hi = mid;
  }
  a = nd[lo < 0 ? 0 : lo];
  return lo;
}

__device__ __forceinline__ double central_root64(const Table64& T, const Star& s) {
  double rmin = div_rn(s.J, sqrt_rn(scale_up<1>(s.E - *T.phi)));
  if (!(rmin >= 0.0)) rmin = 0.0;
  const double r0 = *T.r;
  if (rmin > r0) rmin = r0;
  return rmin;
}

__device__ __forceinline__ int64_t bisect_rmax64(const Table64& T, const Star& s) {
  int64_t lo = s.k, hi = T.nb;
  while (hi - lo > 1) {
    int64_t mid = lo + ((hi - lo) >> 1);
    if (Q_node64(T, s, mid) < 0.0) hi = mid; else lo = mid;
  }
  return lo;
}

__device__ __forceinline__ int64_t bisect_rmin64(const Table64& T, const Star& s) {
  int64_t lo = -1, hi = s.k;
  while (hi - lo > 1) {
    int64_t mid = lo + ((hi - lo) >> 1);
    if (Q_node64(T, s, mid) < 0.0) lo = mid; else hi = mid;
  }
  return lo;
}

// g(s) with Phi from the FP64 table
__device__ __forceinline__ double g64(const Table64& T, const Star& st, double c0, double c1,
                                      double s, double& rs, double& ph, double& Q, int64_t& i) {
  rs = c0 + c1 * (s * (3.0 - s * s));
  const double drds = (3.0 * c1) * (1.0 - s * s);
  i = shell_of(T, rs);
  ph = phi_in_shell(T, i, rs);
  const double L = div_rn(st.J, rs);
  Q = scale_up<1>(st.E - ph) - L * L;
  if (!(Q > 0.0)) return 0.0;
  return div_rn(drds, sqrt_rn(Q));
}

// ------------------------------------------------------------ FP32 side
// sample points of the bound F: s_j = -1 + (j + 1/2)/10.5 (IEEE double,
// evaluated at compile time), and their float roundings
#define CMC_SJ(j) (-1.0 + ((double)(j) + 0.5) / 10.5)
#define CMC_SJ21(f) f(0), f(1), f(2), f(3), f(4), f(5), f(6), f(7), f(8), f(9), f(10), \
    f(11), f(12), f(13), f(14), f(15), f(16), f(17), f(18), f(19), f(20)
__constant__ double c_s64[21] = {CMC_SJ21(CMC_SJ)};
// for the FP32 envelope: s_j (3 - s_j^2) and 3 (1 - s_j^2), rounded to float
#define CMC_SJA(j) ((float)(CMC_SJ(j) * (3.0 - CMC_SJ(j) * CMC_SJ(j))))
#define CMC_SJB(j) ((float)(3.0 * (1.0 - CMC_SJ(j) * CMC_SJ(j))))
__constant__ float c_sa32[21] = {CMC_SJ21(CMC_SJA)};
__constant__ float c_sb32[21] = {CMC_SJ21(CMC_SJB)};

// Radius-bucket index of one segment's float table.  It covers the nodes
// lo..hi, all but the sparse 1/1024 at each end (where a bucket resolution
// fine enough for the core would leave long runs of empty buckets).
// Bucket of a key x > 0: (base - bits(x)) >> shift, base = bits(x_lo).
// Positive floats order like their bit patterns, so buckets are
// non-decreasing along the (non-increasing) keys.  start[b] is the first
// node whose bucket is >= b, start[nbk] = nb.  A node before start[b] has a
// key above any query of bucket b, a node from start[b+1] on (within lo..hi)
// a key below it, so the answer of a query of bucket b lies in
// [start[b] - 1, start[b+1] - 1]; queries above x_lo search [-1, lo),
// queries below x_hi search [hi, nb).
struct Buckets {
  const int* start;
  uint32_t base;
  int shift, nbk, lo, hi;
};

// The shell of the float key xq, to about one node: by the place of the key in
// its bucket (the keys in a bucket are close to uniform), by bisection in the
// tails outside the index.  One look at the index and none at the nodes: every
// caller walks to the exact node from there, and on this GPU the kernels that
// do are bound by the number of random accesses when the tables exceed the L2
// (about 47 G/s).
// K queries at once, so that their looks at the index overlap.
template <int K>
__device__ __forceinline__ void near_shells(const double4_32a* nd, int nb,
                                            const Buckets& B, const float (&xq)[K],
                                            int (&out)[K]) {
  int s0[K], s1[K];
#pragma unroll
  for (int q = 0; q < K; ++q) {
    const long long d = (long long)B.base - (long long)__float_as_uint(xq[q]);
    const long long b = d >> B.shift;
    s0[q] = s1[q] = -1;
    if (d >= 0 && b < B.nbk && CMC_IN(b + 1, B.nbk + 1)) {
      s0[q] = B.start[b];
      s1[q] = B.start[b + 1];
    }
  }
#pragma unroll
  for (int q = 0; q < K; ++q) {
    const uint32_t d = B.base - __float_as_uint(xq[q]);
    if (s1[q] >= 0) {
      const uint32_t f = B.shift ? d << (32 - B.shift) : 0u;  // 2^32 x the place
      out[q] = s0[q] - 1 +
               (int)(((unsigned long long)(uint32_t)(s1[q] - s0[q]) * f + 0x80000000ull) >> 32);
    } else {
      const bool inner = (long long)B.base < (long long)__float_as_uint(xq[q]);
      const long long kq = dbits((double)xq[q]);  // (positive doubles order like their bits)
      int lo = inner ? -1 : B.hi, hi = inner ? B.lo : nb;
      while (hi - lo > 1) {
        const int m = lo + ((hi - lo) >> 1);
        if (dbits(nd[m].x) >= kq) lo = m; else hi = m;
      }
      out[q] = lo;
    }
  }
}

// The potential grid of one segment (see BucketArgs): Phi (float) at the
// float keys key0 + g 2^sh of 1/r.  Inside a binade a float's key is linear
// in its value, so on a binade-aligned grid Phi, linear in 1/r between
// stars, is interpolated linearly in the key up to the kinks of the stars
// inside one cell (relative error ~2e-7 at 1024 cells per binade).
struct Grid {
  const float* phi;
  uint32_t key0, kmax;
  int sh, cells;
  float phi0, mb, x0, err;  // err: relative bound on the interpolation error
};

__device__ __forceinline__ Grid grid_of(const BucketArgs& B, int c) {
  Grid G;
  const int4 pr = B.gprm[c];
  const float4 au = B.gaux[c];
  G.phi = B.gphi + B.goff[c];
  G.key0 = (uint32_t)pr.x;
  G.sh = pr.y;
  G.cells = pr.z;
  G.kmax = (uint32_t)pr.w;
  G.phi0 = au.x;
  G.mb = au.y;
  G.x0 = au.z;
  G.err = au.w;
  return G;
}

__device__ __forceinline__ float grid_phi(const Grid& G, float xq) {
  const uint32_t key = __float_as_uint(xq);
  if (key >= G.kmax) return G.phi0;                               // inside the first star
  if (key < G.key0) return *G.phi + G.mb * (G.x0 - xq);     // beyond the last
  const uint32_t d = key - G.key0;
  const int g = (int)(d >> G.sh);
  if (!CMC_IN(g + 1, G.cells)) return G.phi0;
  // f = (d mod 2^sh) 2^-sh, exact: 1 + f assembled from its bits, minus 1
  const float f =
      __uint_as_float(0x3F800000u | ((d & ((1u << G.sh) - 1u)) << (23 - G.sh))) - 1.0f;
  const float a = G.phi[g], b = G.phi[g + 1];
  return a + f * (b - a);
}

// g(s_j) = (dr/ds) / sqrt(Q) at envelope sample j in FP32 with Phi from the
// grid (sa = s(3 - s^2), sb = 3 (1 - s^2) from the tables).  The envelope
// F = 1.2 max_j g(s_j) only has to bound g: the reciprocal and the inverse
// square root are the one-instruction approximations (relative errors
// below 2^-22), far inside the factor 1.2.
__device__ __forceinline__ float g32_grid(const Grid& G, float E, float J, float c0, float c1,
                                          float sa, float sb) {
  const float rs = c0 + c1 * sa;
  const float drds = c1 * sb;
  float xq, rq;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(xq) : "f"(rs));
  const float ph = grid_phi(G, xq);
  const float L = J * xq;
  const float Q = 2.0f * (E - ph) - L * L;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rq) : "f"(Q));
  return Q > 0.0f ? drds * rq : 0.0f;
}

// about the shell of the point r(s) (bucket index), the start of the FP64
// shell walk of an accepted or edge point
__device__ __forceinline__ int shell32_of(const double4_32a* nd, int nb,
                                          const Buckets& B, float c0, float c1, float sv) {
  const float rs = c0 + c1 * (sv * (3.0f - sv * sv));
  float xq;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(xq) : "f"(rs));
  const float q[1] = {xq};
  int sh[1];
  near_shells<1>(nd, nb, B, q, sh);
  return sh[0];
}

// Mixed mode: the orbit point r(s) in FP64 from an FP32 shell index sh
// (moved to the exact shell), Phi from the enclosed-mass slope of its
// shell (Eq. 6: Phi = Phi_i + M_i (1/r_i - 1/r)), L = J / r and Q.
__device__ __forceinline__ void point64(const double4_32a* nd, int64_t nb,
                                        const Star& st, double c0, double c1, double sv, int sh,
                                        double& rs, double& xs, double& ph, double& L,
                                        double& Q, int& i64) {
  rs = c0 + c1 * (sv * (3.0 - sv * sv));
  double4_32a a;
  i64 = (int)fix_shell_nodes(nd, nb, sh, rs, a);
  xs = div_rn(1.0, rs);
  ph = i64 < 0 ? a.y : a.y + a.w * (a.x - xs);
  L = st.J * xs;
  Q = scale_up<1>(st.E - ph) - L * L;
}


// FP64 mode: the orbit point r(s) in FP64 from an FP32 shell guess sh
// (moved to the exact shell), Phi by Eq. 6's division form (the FP64
// statement of the method, as phi_in_shell), L = J / r and Q.
// sa = s (3 - s^2), the factor of c1 in r(s) (a table entry at the
// envelope's samples)
__device__ __forceinline__ void point64_div_sa(const double4_32a* nd, int64_t nb,
                                               const Star& st, double c0, double c1, double sa,
                                               int sh, double& rs, double& ph, double& Q,
                                               double& L, double& xq, int& i) {
  rs = c0 + c1 * sa;
  double4_32a a;
  i = (int)fix_shell_nodes(nd, nb, sh, rs, a);
  xq = div_rn(1.0, rs);
  if (i < 0) {
    ph = a.y;  // node 0's Phi: the central constant
  } else {
    double xj1 = 0.0, pj1 = 0.0;
    if (i + 1 < nb) {
      const double4_32a b = nd[i + 1];
      xj1 = b.x;
      pj1 = b.y;
    }
    const double den = a.x - xj1;
    ph = !(den > 0.0) ? a.y : a.y + div_rn(a.x - xq, den) * (pj1 - a.y);
  }
  L = div_rn(st.J, rs);
  Q = scale_up<1>(st.E - ph) - L * L;
}

__device__ __forceinline__ void point64_div(const double4_32a* nd, int64_t nb,
                                            const Star& st, double c0, double c1, double sv,
                                            int sh, double& rs, double& ph, double& Q,
                                            double& L, double& xq, int& i) {
  point64_div_sa(nd, nb, st, c0, c1, sv * (3.0 - sv * sv), sh, rs, ph, Q, L, xq, i);
}

// g(s) of FP64 mode at the point of point64_div, sb = 1 - s^2
__device__ __forceinline__ double g_of_point_sb(double c1, double sb, double Q) {
  if (!(Q > 0.0)) return 0.0;
  return div_rn((3.0 * c1) * sb, sqrt_rn(Q));
}

__device__ __forceinline__ double g_of_point(double c1, double sv, double Q) {
  return g_of_point_sb(c1, 1.0 - sv * sv, Q);
}

// (2k + 1) 2^-24 from the top 23 bits of a word: exact in float, in (0, 1)
__device__ __forceinline__ float u01f(uint32_t hi) {
  // 1 + k 2^-23 assembled from its bits, minus 1 (exact), plus 2^-24
  // (exact): no int -> float conversion
  return (__uint_as_float(0x3F800000u | (hi >> 9)) - 1.0f) + 0x1p-24f;
}

// ------------------------------------------------------- turning points
// 1/r and Phi of a node, its radius and slope (one 16-byte load each)
__device__ __forceinline__ double2 node_rw(const double4_32a* p) {
  return reinterpret_cast<const double2*>(p)[1];
}

// Q at 1/r = x with Phi = p, the FP64 method's own evaluation
__device__ __forceinline__ double q64_of(const Star& s, double x, double p) {
  const double L = s.J * x;
  return scale_up<1>(s.E - p) - L * L;
}

// Parts of a double as floats, from its bits: the top 24 significand bits in
// [1, 2), and 2^exponent (0 unless within 2^-60 .. 2^60).  No conversion
// instructions: on this GPU they take the FP64 pipe.
__device__ __forceinline__ float top_of(unsigned long long u) {
  return __uint_as_float(0x3F800000u | ((unsigned)(u >> 29) & 0x7FFFFFu));
}
__device__ __forceinline__ float pow2_of(unsigned long long u) {
  const unsigned f = (unsigned)(u >> 52) & 0x7FFu;
  return f - 963u <= 120u ? __uint_as_float((f - 896u) << 23) : 0.0f;
}

// ---- double-float (float pairs): a value as hi + lo with two floats, from
// the error-free sum of two floats (Knuth's two-sum; every operation rounds
// once, no contraction) and product (the fused multiply-add gives the
// product's error exactly).
struct DF {
  float hi, lo;
};

// |v| to 2^-46 of it (its sign bit set in neg) for a double with pow2_of p2 > 0:
// the top 24 significand bits, then the next 23
__device__ __forceinline__ DF df_of(unsigned long long u, float p2) {
  DF d;
  d.hi = top_of(u) * p2;
  d.lo = ((__uint_as_float(0x4B000000u | ((unsigned)(u >> 6) & 0x7FFFFFu)) - 8388608.0f) *
          0x1p-46f) * p2;
  return d;
}

__device__ __forceinline__ DF df_norm(float hi, float lo) {
  const float s = hi + lo;
  DF d;
  d.hi = s;
  d.lo = lo - (s - hi);
  return d;
}

__device__ __forceinline__ DF df_sub(DF a, DF b) {
  const float s = a.hi - b.hi, bb = s - a.hi;
  const float e = (a.hi - (s - bb)) - (b.hi + bb);
  return df_norm(s, e + (a.lo - b.lo));
}

__device__ __forceinline__ DF df_mul(DF a, DF b) {
  const float p = a.hi * b.hi;
  const float e = __fmaf_rn(a.hi, b.hi, -p);
  return df_norm(p, e + (a.hi * b.lo + a.lo * b.hi));
}

// The star's constants of the walks below: |E|, J as float pairs (E < 0), J^2
struct WalkStar {
  DF E, J;
  float J2;
  bool ok;  // both within the float pairs' range
};

// The node of a sign change of Q, by a walk from node p (lo <= p <= hi; 1/r = x, Phi
// = ph there).  Q counts as >= 0 at the star's end (at_hi false: r_max, whose star
// is lo; true: r_min, whose star is hi) and as < 0 at the other end.  Returns
// the lower node of the pair with different signs, -2 when the walk is too long.
// Every sign is that of the FP64 method's evaluation of Q, found in floats:
//
// At p, Q = 2 (|Phi| - |E|) - (J x)^2 in float pairs.  E, J, 1/r and Phi are within
// 2^-46, each pair sum adds at most 2^-46 of its operands and each pair
// product 2^-45 of its result, so Q is within 2^-41.5 of S = |E| + |Phi| + L^2; the
// FP64 evaluation is within 2^-50 S.  Beyond 2^-40 S the sign is certain.
//
// A node near p has Q = Q_p + 2 (|Phi| - |Phi_p|) - J^2 (x + x_p) (x - x_p).  In p's
// binades the differences are those of the significands' bits (the top 24
// exactly, the rest to 2^-44), J^2 is within 2^-22, x + x_p and each operation
// round to 2^-24, Q_p to 2^-24 |Q_p| <= 2^-24 (|Q| + T), T the two terms'
// magnitudes: within 2^-20 T + 2^-22 |Q| + 2^-41 S in all, and S there at most S + T.
// Beyond 2^-19 T + 2^-40 S the sign is certain: 25 instructions.
//
// Otherwise the FP64 evaluation decides.
struct Bracket {
  int j;        // the lower node; -1: inside node 0, whose values it then has
  double x, p;  // its 1/r and Phi
};

__device__ __forceinline__ bool walk_sign(const Star& s, const WalkStar& W,
                                          const double4_32a* nd, int nb, int p,
                                          int lo, int hi, bool at_hi, double2 at, Bracket& B) {
  const unsigned long long xb = ubits(at.x), pb = ubits(at.y);
  const float ex = pow2_of(xb), ep = pow2_of(pb);
  const bool ok = W.ok && ex * ep != 0.0f;
  const float x1 = top_of(xb), p1 = top_of(pb), x0 = x1 * ex;
  const DF P = df_of(pb, ep), L = df_mul(W.J, df_of(xb, ex)), L2 = df_mul(L, L);
  const DF d = df_sub(P, W.E), q2 = df_sub(DF{2.0f * d.hi, 2.0f * d.lo}, L2);
  const float q0 = q2.hi != 0.0f ? q2.hi : q2.lo;
  const float s40 = 0x1p-40f * ((W.E.hi + P.hi) + L2.hi);
  bool pos = p == (at_hi ? hi : lo);
  if (!pos && p != (at_hi ? lo : hi))
    pos = ok && fabsf(q0) > s40 ? q0 > 0.0f : !lt0(q64_of(s, at.x, at.y));
  const int step = pos == at_hi ? -1 : 1;
  for (int w = 0; w < 64; ++w) {
    const int c = p + step;
    bool now = (c >= hi) == at_hi;
    double2 t = at;
    if (c >= 0 && c < nb) t = node_xp(nd + c);
    if (c > lo && c < hi) {
      const unsigned long long xcb = ubits(t.x), pcb = ubits(t.y);
      // the differences of the low 29 bits, to 2^8 of them
      const int lx = ((int)((unsigned)xcb & 0x1FFFFFFFu) - (int)((unsigned)xb & 0x1FFFFFFFu)) >> 8;
      const int lp = ((int)((unsigned)pcb & 0x1FFFFFFFu) - (int)((unsigned)pb & 0x1FFFFFFFu)) >> 8;
      const float fx = __uint_as_float(0x4B400000u + (unsigned)lx) - 12582912.0f;
      const float fp = __uint_as_float(0x4B400000u + (unsigned)lp) - 12582912.0f;
      const float dx = __fmaf_rn(fx, 0x1p-44f, top_of(xcb) - x1) * ex;
      const float a = 2.0f * (__fmaf_rn(fp, 0x1p-44f, top_of(pcb) - p1) * ep);
      const float b = (W.J2 * (2.0f * x0 + dx)) * dx;
      const float q = (q0 + a) - b;
      const bool sure = ok && (((xcb ^ xb) | (pcb ^ pb)) >> 52) == 0ull &&
                        fabsf(q) > __fmaf_rn(0x1p-19f, fabsf(a) + fabsf(b), s40);
      now = q > 0.0f;
      if (!sure) now = !lt0(q64_of(s, t.x, t.y));
    }
    if (now != pos) {
      B.j = step > 0 ? p : c;
      B.x = step > 0 ? at.x : t.x;
      B.p = step > 0 ? at.y : t.y;
      return true;
    }
    p = c;
    at = t;
  }
  return false;
}

// Q in FP32 at grid point g (1/r from the grid key, Phi from the grid)
__device__ __forceinline__ float grid_q(const Grid& G, float E, float J2, int g, float& xg) {
  xg = __uint_as_float(G.key0 + ((uint32_t)g << G.sh));
  return __fmaf_rn(-J2 * xg, xg, 2.0f * (E - G.phi[g]));
}

// Node brackets of both turning points: r_max's node j with Q >= 0 (the star
// k counts as such) and j + 1 with Q < 0 (or the virtual node nb), r_min's j with
// Q < 0 (or -1) and j + 1 with Q >= 0 (or the star).  The sign changes of Q on
// the grid points (both searches abreast, a fixed number of rounds on a grid
// that stays in the L1), the root inside the cell by linear interpolation in
// 1/r, its node through the bucket index, and a walk from there to where the
// FP64 evaluation of Q changes sign.  Q is concave in 1/r (Phi is convex), so
// that sign change is the only one on its side and the search before the walk
// need not be exact, only close.  False when a walk is too long.
//
// Bound by the L1's gathers (one wavefront per lane; 60-69% busy) with the FP64
// pipe half busy.  N = 1e7: 0.99 ms, 180 B of DRAM a star; with a float-pair copy
// of the table for the searches and walks, probes of four nodes a round and
// FP64 walks where uncertified 1.27 ms, 338 B.  Both walks in one loop (1.08),
// four-way grid rounds (1.08), the grid's top levels in shared memory (1.01)
// and 40 to 64 registers (0.98 to 1.01) gave nothing.
__device__ __forceinline__ bool grid_brackets(const Grid& G, const double4_32a* nd,
                                              const Buckets& BK, const Star& s, int nb, int k,
                                              float xk, float qk, Bracket& bmax,
                                              Bracket& bmin) {
  WalkStar W;
  const float pE = pow2_of(ubits(s.E)), pJ = pow2_of(ubits(s.J));
  W.ok = pE * pJ != 0.0f;
  W.E = df_of(ubits(s.E), pE);
  W.J = df_of(ubits(s.J), pJ);
  W.J2 = W.J.hi * W.J.hi;
  // (out of the pairs' range: radial or all but unbound orbits)
  const float E = W.ok ? -W.E.hi : f32_rn(s.E);
  const float J2 = W.ok ? W.J2 : f32_rn(s.J) * f32_rn(s.J);
  const uint32_t kk = __float_as_uint(xk);
  if (G.cells < 2 || kk < G.key0) return false;
  int gk = (int)((kk - G.key0) >> G.sh);  // grid points 0..gk lie at or outside the star
  if (gk > G.cells - 1) gk = G.cells - 1;
  // r_max: the last grid point in [0, gk] with Q < 0 (-1: none; Q -> 2E < 0 as 1/r -> 0)
  // r_min: the last one in [gk + 1, cells) with Q >= 0 (gk: none)
  int ga = -1, gb = gk;
  for (int st = 1 << (31 - __clz(G.cells)); st > 0; st >>= 1) {
    const int ma = ga + st, mb = gb + st;
    float x;
    const float qa = grid_q(G, E, J2, ma < gk ? ma : gk, x);
    const float qb = grid_q(G, E, J2, mb < G.cells ? mb : G.cells - 1, x);
    if (ma <= gk && qa < 0.0f) ga = ma;
    if (mb < G.cells && !(qb < 0.0f)) gb = mb;
  }
  // root estimates between the two points of each sign change (the star itself
  // on its side of the grid), and their nodes
  const bool none1 = ga < 0, none2 = gb + 1 >= G.cells;
  float xq[2];
  {
    float xl, xh;
    const float ql = grid_q(G, E, J2, none1 ? 0 : ga, xl);
    float qh = grid_q(G, E, J2, ga == gk ? gk : ga + 1, xh);
    if (ga == gk) {
      xh = xk;
      qh = qk;
    }
    xq[0] = xl + (xh - xl) * __fdividef(ql, ql - qh);
  }
  {
    float xl, xh;
    float ql = grid_q(G, E, J2, gb, xl);
    const float qh = grid_q(G, E, J2, none2 ? gb : gb + 1, xh);
    if (gb == gk) {
      xl = xk;
      ql = qk;
    }
    xq[1] = xl + (xh - xl) * __fdividef(ql, ql - qh);
  }
  int pn[2];
  near_shells<2>(nd, nb, BK, xq, pn);
  int p1 = none1 ? nb - 1 : pn[0], p2 = none2 ? -1 : pn[1];
  p1 = p1 < k ? k : (p1 > nb - 1 ? nb - 1 : p1);
  p2 = p2 < -1 ? -1 : (p2 > k - 1 ? k - 1 : p2);
  const int i2 = p2 < 0 ? 0 : p2;
  const double2 t1 = node_xp(nd + p1), t2 = node_xp(nd + i2);
  return walk_sign(s, W, nd, nb, p1, k, nb, false, t1, bmax) &&
         walk_sign(s, W, nd, nb, p2, -1, k, true, t2, bmin);
}

// Mixed mode, turning points of one bound star with E < 0: the brackets on the
// grid and the nodes, or where a walk gives up by FP64 bisection, then the FP64
// roots inside the bracketing shells (Eq. 12).
__device__ __forceinline__ void turning_mixed(const Table64& T,
                                              const double4_32a* nd, const Grid& G,
                                              const Buckets& BK, const Star& s, float xk,
                                              float qk, double& rmin, double& rmax) {
  const int nb = (int)T.nb, k = (int)s.k;
  Bracket a, b;
  if (!grid_brackets(G, nd, BK, s, nb, k, xk, qk, a, b)) {
    a.j = (int)bisect_rmax64(T, s);
    b.j = (int)bisect_rmin64(T, s);
    const double2 ta = node_xp(nd + a.j), tb = node_xp(nd + (b.j < 0 ? 0 : b.j));
    a.x = ta.x;
    a.p = ta.y;
    b.x = tb.x;
    b.p = tb.y;
  }
  const double2 ra = node_rw(nd + a.j), rb = node_rw(nd + (b.j < 0 ? 0 : b.j));
  const double r1 = nd[a.j + 1 < nb ? a.j + 1 : a.j].z, r2 = nd[b.j + 1].z;
  rmax = rmax_core(s, ra.x, a.x, a.p, ra.y, a.j + 1 < nb, r1);
  rmin = rmin_core(s, b.j < 0, rb.x, b.x, b.p, b.j < 0 ? 0.0 : rb.y, b.j >= 0, r2);
}

// First kernel of the mixed-mode orbit step: the turning points of every
// bound star with E < 0, into tp_min / tp_max (split from the sampling
// kernel so that each runs with fewer registers and more warps).
template <int kMinB>
__global__ void __launch_bounds__(256, kMinB) k_turning_mixed(
    Seg S, const double* r, const double* x, const double* phi,
    const double* vr, const double* vt, BucketArgs BA, double* tp_min,
    double* tp_max, double4_32a* orb, int64_t n) {
  pdl_enter();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const int c = seg_find(S.off, S.n_seg, p);
  const int64_t sb = S.off[c];
  const int64_t nbc = S.nb[c];
  const int64_t k = p - sb;
  if (k >= nbc) return;
  const Table64 T{r + sb, x + sb, phi + sb, nbc};
  const double rk = r[p], vrk = vr[p], vtk = vt[p];
  Star s;
  s.k = k;
  s.E = T.phi[k] + scale_down<1>(vrk * vrk + vtk * vtk);
  s.J = rk * vtk;
  // E < 0 on the bit pattern (negative, nonzero, not NaN); otherwise an
  // escaper, which the sampling kernel handles
  const unsigned long long eb = ubits(s.E);
  if (!(eb > 0x8000000000000000ull && eb <= 0xFFF0000000000000ull)) {
    orb[p] = make_double4_32a(s.E, s.J, 0.0, 0.0);
    return;
  }
  double rmin, rmax;
  Buckets BK;
  const int4 pr = BA.prm[c];
  BK.start = BA.start + BA.off[c];
  BK.base = BA.base[c];
  BK.shift = pr.x;
  BK.nbk = pr.y;
  BK.lo = pr.z;
  BK.hi = pr.w;
  // (Q at the star is v_r^2; its 1/r only has to place it on the grid)
  const float vr32 = f32_rn(vrk);
  float xk;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(xk) : "f"(f32_rn(rk)));
  turning_mixed(T, BA.node + sb, grid_of(BA, c), BK, s, xk, vr32 * vr32, rmin, rmax);
  if (tp_min) {
    tp_min[p] = rmin;
    tp_max[p] = rmax;
  }
  // the orbit's record for the sampling kernels: E, J, c0 = (r_max + r_min)
  // / 2 and c1 = (r_max - r_min) / 4 (c1 > 0 exactly when r_max > r_min:
  // radii are far from the underflow range)
  orb[p] = make_double4_32a(s.E, s.J, scale_down<1>(rmax + rmin), scale_down<2>(rmax - rmin));
}

// One trial's accept test in FP32 with a bound on its error: +1 accepted,
// 0 rejected, -1 undecided (the trial is then taken in FP64).  The test is
// F X' < g(s), g = (dr/ds) / sqrt(Q), at the FP64 point s (52 bits) and
// X' (53 bits); the float values use 23 bits of each, so |s32 - s| and
// |X'32 - X'| are at most 2^-23 and 2^-24.  Bounds (u = 2^-24):
//   r(s):  |r32 - r| <= 3|c1| (1 - s^2 + 2^-21) 2^-23 + 8u (|c0| + 2|c1|)
//          + 2^-22 |r|                         1/r by the approximate reciprocal
//   Q:     16u (|E| + |Phi| + L^2)             float operations and inputs
//          + (2 err_grid + 4u) |Phi|           grid interpolation and values
//          + 1.5 * 2 (M x + L^2) |dr| / r      Q's slope in r, M <= M_bound
//   g:     1.5 * (1/2) dQ / Q + 6|c1| 2^-23 / (dr/ds) + 16u
//          + 2^-21                             the approximate 1/sqrt(Q)
// Close to a turning point Q is within a few dQ of zero and the trial is
// left undecided; elsewhere the FP32 answer is the FP64 one.
// kExact (FP64 mode): F is the float of the FP64 envelope, and a trial
// whose g might lie on either side of F is left undecided too, so that the
// count of g > F (violations) is the FP64 one.
template <bool kExact>
__device__ __forceinline__ int accept32(const Grid& G, float E, float J, float c0, float c1,
                                        float F, float sv, float xp,
                                        unsigned long long& viol) {
  const float ss = sv * sv;
  const float rs = c0 + c1 * (sv * (3.0f - ss));
  const float drds = (3.0f * c1) * (1.0f - ss);
  // the one-instruction reciprocal and inverse square root (relative
  // errors below 2^-22): the reciprocal's error counts as an error in r (in
  // dr), the inverse square root's in eg (2^-21), and eg, computed with them,
  // is taken 2^-16 larger
  float xq;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(xq) : "f"(rs));
  const float ph = grid_phi(G, xq);
  const float L = J * xq, L2 = L * L;
  const float Q = 2.0f * (E - ph) - L2;
  const float ac1 = fabsf(c1), aph = fabsf(ph);
  const float dr = 3.0f * ac1 * ((1.0f - ss) + 0x1p-21f) * 0x1p-23f +
                   0x1p-21f * (fabsf(c0) + 2.0f * ac1) + 0x1p-22f * fabsf(rs);
  const float qerr = 0x1p-20f * (fabsf(E) + aph + L2) + (2.0f * G.err + 0x1p-22f) * aph +
                     3.0f * (G.mb * xq + L2) * (dr * xq);
  if (!(Q > 4.0f * qerr) || !(drds > 0x1p-100f)) return -1;
  float rq, rd;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rq) : "f"(Q));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rd) : "f"(drds));
  const float g = drds * rq;
  const float eg = ((0.75f * qerr) * (rq * rq) + (6.0f * ac1 * 0x1p-23f) * rd + 0x1p-20f +
                    0x1p-21f) * (1.0f + 0x1p-16f);
  if (!(eg < 0.25f)) return -1;
  if (kExact) {
    const bool above = g * (1.0f - eg) > F * (1.0f + 0x1p-22f);
    const bool below = g * (1.0f + eg) < F * (1.0f - 0x1p-22f);
    if (!above && !below) return -1;
  }
  const float a = F * xp, da = F * 0x1p-22f;
  if (a + da < g * (1.0f - eg)) {
    if (g > F) ++viol;
    return 1;
  }
  if (a - da > g * (1.0f + eg)) {
    if (g > F) ++viol;
    return 0;
  }
  return -1;
}

// g(s) in FP32 at an envelope sample with the error bound of accept32
// (the sample's float s is within 2^-25 of the FP64 one): 1 with g and its
// relative bound eg, 0 when Q < 0 for certain (g = 0), -1 when FP32 cannot
// tell.  The reciprocal and the inverse square root are the one-instruction
// approximations (relative errors below 2^-22): the reciprocal's error is an
// error in r (added to dr, as r's own), the inverse square root's goes into
// eg (2^-21), and eg itself, computed with them, is taken 2^-16 larger.
__device__ __forceinline__ int g32_bounded(const Grid& G, float E, float J, float c0, float c1,
                                           float sv, float& g, float& eg) {
  const float ss = sv * sv;
  const float rs = c0 + c1 * (sv * (3.0f - ss));
  const float drds = (3.0f * c1) * (1.0f - ss);
  float xq;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(xq) : "f"(rs));
  const float ph = grid_phi(G, xq);
  const float L = J * xq, L2 = L * L;
  const float Q = 2.0f * (E - ph) - L2;
  const float ac1 = fabsf(c1), aph = fabsf(ph);
  const float dr = 3.0f * ac1 * ((1.0f - ss) + 0x1p-21f) * 0x1p-23f +
                   0x1p-21f * (fabsf(c0) + 2.0f * ac1) + 0x1p-22f * fabsf(rs);
  const float qerr = 0x1p-20f * (fabsf(E) + aph + L2) + (2.0f * G.err + 0x1p-22f) * aph +
                     3.0f * (G.mb * xq + L2) * (dr * xq);
  if (Q < -4.0f * qerr) return 0;
  if (!(Q > 4.0f * qerr) || !(drds > 0x1p-100f)) return -1;
  float rq, rd;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rq) : "f"(Q));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rd) : "f"(drds));
  g = drds * rq;
  eg = ((0.75f * qerr) * (rq * rq) + (6.0f * ac1 * 0x1p-23f) * rd + 0x1p-20f + 0x1p-21f) *
       (1.0f + 0x1p-16f);
  if (!(eg < 0.25f)) return -1;
  return 1;
}

// the envelope samples s_j as floats (within 2^-25 of the FP64 ones)
#define CMC_SJF(j) ((float)CMC_SJ(j))
__constant__ float c_s32[21] = {CMC_SJ21(CMC_SJF)};

// FP64 mode's envelope F = 1.2 max_j g(s_j) over the 21 samples, the FP64
// value (Eq. 6's division form, as the FP64 statement of the method):
// every g(s_j) is first bounded in FP32 (g32_bounded); only the samples
// whose upper bound reaches the largest lower bound, and those FP32 cannot
// bound, can hold the maximum, and only they are evaluated in FP64.  Nearly
// circular orbits have a flat g and FP32 bounds too loose to rank their
// samples, so the candidates per star range from 1 to 21 (about 1.1 on
// average).  Two kernels: k_env_screen bounds the samples and lists the
// candidate (star, sample) pairs; k_env_eval evaluates them one pair per
// thread (whole warps busy, where one warp pooling its own stars' pairs
// left most lanes idle in its last round), the maximum per star kept in
// gmax as bits (g >= 0 orders as its bits).  gmax = 0 for stars without an
// orbit to sample (r_max <= r_min: every g is 0 or negative there); the
// readers take F = 1.2 gmax.
constexpr int kEnvThreads = 128;
constexpr uint64_t kEnvNone = ~0ull;  // a list slot left empty

// s_j (3 - s_j^2) and 1 - s_j^2 at the 21 samples, computed once on the
// device with the operations of point64_div and g_of_point (k_env_tables)
__device__ double g_env_sa[21], g_env_sb[21];

__global__ void k_env_tables() {
  pdl_enter();
  const int j = threadIdx.x;
  if (j >= 21) return;
  const double sv = c_s64[j];
  g_env_sa[j] = sv * (3.0 - sv * sv);
  g_env_sb[j] = 1.0 - sv * sv;
}

// FP64 g at sample j of a star (one copy for the list and the spill loops)
__device__ __noinline__ double g64_sample(const double4_32a* nd, int64_t nb,
                                          const Buckets& BK, double E, double J, double c0,
                                          double c1, int j) {
  Star s;
  s.k = 0;
  s.E = E;
  s.J = J;
  const float c0f = f32_rn(c0), c1f = f32_rn(c1);
  double rs, ph, Q, L, xq;
  int i;
  point64_div_sa(nd, nb, s, c0, c1, g_env_sa[j],
                 shell32_of(nd, (int)nb, BK, c0f, c1f, c_s32[j]), rs, ph, Q, L, xq, i);
  return g_of_point_sb(c1, g_env_sb[j], Q);
}

__device__ __forceinline__ Buckets buckets_of(const BucketArgs& BA, int c) {
  Buckets BK;
  const int4 pr = BA.prm[c];
  BK.start = BA.start + BA.off[c];
  BK.base = BA.base[c];
  BK.shift = pr.x;
  BK.nbk = pr.y;
  BK.lo = pr.z;
  BK.hi = pr.w;
  return BK;
}

// E, J and the orbit's c0 = (r_max + r_min) / 2, c1 = (r_max - r_min) / 4
// of star p (segment c) from the turning-point kernel's record; false where
// there is no orbit to sample
__device__ __forceinline__ bool env_star(const Seg& S, const double4_32a* orb, int64_t p,
                                         int& c, double& E, double& J, double& c0, double& c1) {
  c = seg_find(S.off, S.n_seg, p);
  const int64_t nbc = S.nb[c], k = p - S.off[c];
  if (!(k < nbc)) return false;
  const double4_32a o = orb[p];
  E = o.x;
  J = o.y;
  c0 = o.z;
  c1 = o.w;
  return lt0(E) && gt_pos(c1, 0.0);
}

// kG > 1 (few stars, as k_sample32): kG lanes a star share the samples.  FP64 mode's
// orbit stage of 10^3, 10^4, 3 x 10^4 stars 43.0, 45.4, 47.9 us with a lane a star here,
// 33.9, 34.3, 40.3 so (2 to 3 us of it two fills less).
template <int kG>
__global__ void __launch_bounds__(kEnvThreads) k_env_screen(Seg S, BucketArgs BA,
                                                            const double4_32a* orb, EnvWork W,
                                                            int64_t n) {
  pdl_enter();
  __shared__ float s_hi[21][kEnvThreads];  // upper bounds of the samples
  const int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kG;
  const int lane = threadIdx.x & 31, sub = lane & (kG - 1);
  const unsigned group = ((kG == 32 ? 0u : 1u << kG) - 1u) << (lane - sub);
  int c = -1;
  unsigned cand = 0u;
  if (p < n) {
    double E, J, c0, c1;
    if (env_star(S, orb, p, c, E, J, c0, c1)) {
      // the star's values for the evaluation of its pairs
      if (sub == 0) W.star[p] = make_double4_32a(E, J, c0, c1);
      const float c0f = f32_rn(c0), c1f = f32_rn(c1), E32 = f32_rn(E), J32 = f32_rn(J);
      const Grid GD = grid_of(BA, c);
      unsigned pos = 0u;
      float lo_max = 0.0f;
      // one copy of the sample code (not unrolled: code size), the upper
      // bounds kept in shared memory
#pragma unroll 1
      for (int jj = sub; jj < 21; jj += kG) {
        float g = 0.0f, eg = 0.0f;
        const int st = g32_bounded(GD, E32, J32, c0f, c1f, c_s32[jj], g, eg);
        float h = 0.0f;
        if (st > 0) {
          const float lo = g * (1.0f - eg);
          h = g * (1.0f + eg);
          lo_max = lo > lo_max ? lo : lo_max;
          pos |= 1u << jj;
        } else if (st < 0) {
          cand |= 1u << jj;
        }
        s_hi[jj][threadIdx.x] = h;
      }
      // (bits of floats >= 0 order like them)
      if (kG > 1) lo_max = __uint_as_float(__reduce_max_sync(group, __float_as_uint(lo_max)));
#pragma unroll 1
      for (int jj = sub; jj < 21; jj += kG)
        if (((pos >> jj) & 1u) && s_hi[jj][threadIdx.x] >= lo_max) cand |= 1u << jj;
      if (kG > 1) {
        cand = __reduce_or_sync(group, cand);
        if (sub != 0) cand = 0u;  // the star's pairs are its first lane's
      }
    }
    if (sub == 0) W.gmax[p] = 0.0;
  }
  // the warp's pairs go to the list in lane order, with one atomic
  const unsigned cnt = (unsigned)__popc(cand);
  unsigned incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += v;
  }
  const unsigned total = __shfl_sync(0xFFFFFFFFu, incl, 31);
  if (total) {
    unsigned long long base = 0ull;
    if (lane == 0) base = atomicAdd(W.cnt, (unsigned long long)total);
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    const unsigned long long cap = (unsigned long long)W.cap;
    if (base + total <= cap) {
      unsigned long long at = base + (incl - cnt);
      for (unsigned m = cand; m; m &= m - 1u)
        W.list[at++] = ((uint64_t)p << 5) | (uint64_t)(__ffs(m) - 1);
    } else {
      // the list is full: its slots reserved here stay empty, and the
      // stars go to the spill list (one entry per star, never full)
      for (unsigned long long e = base + lane; e < base + total && e < cap; e += 32)
        W.list[e] = kEnvNone;
      if (cnt) {
        const unsigned long long at = atomicAdd(W.cnt + 1, 1ull);
        W.spill[at] = ((uint64_t)p << 21) | (uint64_t)cand;
      }
    }
  }
  // FP64 evaluations: one atomic per segment present in the warp
  const unsigned am = __ballot_sync(0xFFFFFFFFu, p < n);
  if (p < n) {
    const unsigned peers = __match_any_sync(am, c);
    const unsigned tot = __reduce_add_sync(peers, cnt);
    if (lane == __ffs(peers) - 1) stat_add(S.stats, c, kStEnvelope64, tot);
  }
}

// FP64 g of one listed pair into its star's maximum (E, J, c0, c1 from the
// screening kernel's record of the star)
__device__ __forceinline__ void env_pair(const Seg& S, const BucketArgs& BA, const EnvWork& W,
                                         int64_t p, int jj) {
  const int c = seg_find(S.off, S.n_seg, p);
  const double4_32a v = W.star[p];
  const int64_t sb = S.off[c];
  const Buckets BK = buckets_of(BA, c);
  double* gmax = W.gmax;
  const double g = g64_sample(BA.node + sb, S.nb[c], BK, v.x, v.y, v.z, v.w, jj);
  if (g > 0.0) atomicMax((unsigned long long*)(gmax + p), (unsigned long long)__double_as_longlong(g));
}

__global__ void __launch_bounds__(kEnvThreads) k_env_eval(Seg S, BucketArgs BA, EnvWork W) {
  pdl_enter();
  const unsigned long long cap = (unsigned long long)W.cap;
  const unsigned long long np = W.cnt[0] < cap ? W.cnt[0] : cap;
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long e = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; e < np;
       e += stride) {
    const uint64_t w = W.list[e];
    if (w == kEnvNone) continue;
    env_pair(S, BA, W, (int64_t)(w >> 5), (int)(w & 31u));
  }
  // spilled stars: 32 at a time per warp, each warp pooling their pairs
  const unsigned long long ns = W.cnt[1];
  const int lane = threadIdx.x & 31;
  const unsigned long long warps = stride / 32;
  for (unsigned long long w0 = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) / 32 * 32;
       w0 < ns; w0 += warps * 32) {
    const unsigned long long i = w0 + lane;
    const uint64_t w = i < ns ? W.spill[i] : 0ull;
    const unsigned cand = (unsigned)(w & 0x1FFFFFu);
    const int64_t ps = (int64_t)(w >> 21);
    const unsigned cnt = (unsigned)__popc(cand);
    unsigned incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += v;
    }
    const unsigned total = __shfl_sync(0xFFFFFFFFu, incl, 31);
    for (unsigned t0 = 0; t0 < total; t0 += 32) {
      const unsigned t = t0 + (unsigned)lane;
      // owner: the first lane whose inclusive count exceeds t
      int own = 0;
#pragma unroll
      for (int step = 16; step > 0; step >>= 1) {
        const unsigned v = __shfl_sync(0xFFFFFFFFu, incl, own + step - 1);
        if (v <= t) own += step;
      }
      const unsigned o_incl = __shfl_sync(0xFFFFFFFFu, incl, own);
      const unsigned o_cnt = __shfl_sync(0xFFFFFFFFu, cnt, own);
      const unsigned o_cand = __shfl_sync(0xFFFFFFFFu, cand, own);
      const long long o_p = __shfl_sync(0xFFFFFFFFu, (long long)ps, own);
      if (t < total) {
        const int rank = (int)(t - (o_incl - o_cnt));  // which of the owner's pairs
        env_pair(S, BA, W, (int64_t)o_p, (int)__fns(o_cand, 0u, rank + 1));
      }
    }
  }
}

// Result of the FP32 sampler in a star's key slot: bits 0-29 the trial
// index, 30-31 the status, 32-63 the bits of F (float)
enum : uint32_t { kSmpAccepted = 0, kSmpPending = 1, kSmpDegenerate = 2, kSmpCap = 3 };

// Second kernel of the mixed-mode orbit step (after k_turning_mixed): the
// envelope F = 1.2 max g over the 21 samples with Phi from the potential
// grid, then the FP32 trials (accept32) up to the first one that is
// accepted (kSmpAccepted) or that FP32 cannot decide (kSmpPending:
// k_pending64 takes it and the rest of the sequence in FP64).  Only
// float state is live in the loop, so the kernel runs at full occupancy
// without spilling.  F only has to bound g: 1.2 max g over these FP32
// samples is as valid an envelope as the FP64 one (it differs from it by up
// to ~1e-4 at the outer samples, so the two modes draw different, equally
// exact, accept sequences).
// kExact (FP64 mode): F is FP64 mode's envelope, 1.2 Fx (Fx from k_env_eval),
// and a trial is decided here only where the FP64 decision and violation
// count are certain.
// kG > 1 (few stars, chip idle): kG lanes a star share the envelope's samples and
// take kG trials at a time, the first one that is accepted or undecided counts.
// Orbit stage of 10^3, 10^4, 3 x 10^4, 6 x 10^4 stars 24.9, 29.1, 30.8, 32.9 us with a
// lane, 22.4, 23.8, 26.7, 32.9 with four, 20.4, 22.8, 28.6, 36.3 with eight.
// (The rule is sampler_lanes.)
constexpr int kOwnTrials = 2;

template <int kMinB, bool kTaus, bool kExact, int kG>
__global__ void __launch_bounds__(256, kMinB) k_sample32(Seg S, int max_trials,
                                                  const uint32_t* id,
                                                  const uint32_t* step_p, BucketArgs BA,
                                                  const double4_32a* orb,
                                                  uint64_t* keys, uint32_t* plist,
                                                  uint32_t* pcount, int64_t n, const double* Fx) {
  pdl_enter();
  const int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kG;
  // (kG > 1: the star's lanes)
  const int lane = threadIdx.x & 31, sub = lane & (kG - 1), at = lane - sub;
  const unsigned group = (kG == 32 ? 0u : 1u << kG) - 1u;
  unsigned long long viol = 0;
  bool pend = false;
  int c = -1;  // lanes past the end form their own group below
  // kG == 1, counter draws: the trials by the warp (below)
  constexpr bool kPool = kG == 1 && !kTaus;
  bool live = false;
  float c0f = 0.0f, c1f = 0.0f, E32 = 0.0f, J32 = 0.0f, F32 = 0.0f;
  uint32_t st = kSmpCap, idv = 0u;
  int t = 0;
  if (p < n) {
    c = seg_find(S.off, S.n_seg, p);
    const int64_t k = p - S.off[c];
    // E, J, c0, c1 from the turning-point kernel
    const double4_32a o = k < S.nb[c] ? orb[p] : make_double4_32a(0.0, 0.0, 0.0, 0.0);
    const double E = o.x;
    if (k < S.nb[c] && lt0(E)) {
      const double J = o.y, c0 = o.z, c1 = o.w;
      c0f = f32_rn(c0), c1f = f32_rn(c1), E32 = f32_rn(E), J32 = f32_rn(J);
      const Grid GD = grid_of(BA, c);
      bool degenerate;
      if (kExact) {
        const double F64 = 1.2 * Fx[p];
        F32 = f32_rn(F64);
        degenerate = !gt_pos(c1, 0.0) || !(F64 > 0.0);
      } else {
        float gmax = 0.0f;
#pragma unroll 3
        for (int j = sub; j < 21; j += kG) {
          const float g = g32_grid(GD, E32, J32, c0f, c1f, c_sa32[j], c_sb32[j]);
          gmax = g > gmax ? g : gmax;
        }
        // (bits of floats >= 0 order like them)
        if (kG > 1)
          gmax = __uint_as_float(__reduce_max_sync(group << at, __float_as_uint(gmax)));
        F32 = 1.2f * gmax;
        degenerate = !gt_pos(c1, 0.0) || !(F32 > 0.0f);
      }
      if (degenerate) {
        st = kSmpDegenerate;
      } else if (kPool) {
        idv = id[p];
        live = true;
        // the first trials in the star's lane
        Draws<false> g = draws_of<false>(S, c, idv, *step_p);
        const int own = max_trials < kOwnTrials ? max_trials : kOwnTrials;
        for (; t < own; ++t) {
          const U4 w = g.block(kTagRej, (uint32_t)t);
          const int d = accept32<kExact>(GD, E32, J32, c0f, c1f, F32, 2.0f * u01f(w.y) - 1.0f,
                                         u01f(w.w), viol);
          if (d == 0) continue;
          st = d > 0 ? kSmpAccepted : kSmpPending;
          live = false;
          break;
        }
        if (t >= max_trials) live = false;
      } else {
        Draws<kTaus> g = draws_of<kTaus>(S, c, id[p], *step_p);
        for (; t < max_trials; t += kG) {
          const int mine = t + sub;
          unsigned long long over = 0;
          int d = 0;
          if (kG == 1 || mine < max_trials) {
            const U4 w = g.block(kTagRej, (uint32_t)mine);
            d = accept32<kExact>(GD, E32, J32, c0f, c1f, F32, 2.0f * u01f(w.y) - 1.0f, u01f(w.w),
                                 over);
          }
          if (kG == 1) {
            viol += over;
            if (d == 0) continue;
            st = d > 0 ? kSmpAccepted : kSmpPending;
            break;
          }
          const unsigned acc = (__ballot_sync(group << at, d > 0) >> at) & group;
          const unsigned any = acc | ((__ballot_sync(group << at, d < 0) >> at) & group);
          const int last = any ? __ffs(any) - 1 : kG - 1;
          if (sub <= last) viol += over;
          if (any) {
            st = (acc >> last) & 1u ? kSmpAccepted : kSmpPending;
            t += last;
            break;
          }
        }
        if (kG > 1 && t > max_trials) t = max_trials;
      }
      if (!kPool && sub == 0) {
        keys[p] = ((uint64_t)__float_as_uint(F32) << 32) | ((uint64_t)st << 30) |
                  (uint64_t)(t & 0x3FFFFFFF);
        pend = st == kSmpPending;
      }
      if (kPool) pend = true;  // (a result to write)
    }
  }
  if (kPool) {
    // The further trials, by rounds.  While more than half the lanes are undecided
    // each takes its own star's next one; then the lanes are shared out, G to each
    // star that is left, for its next G trials (stars of one segment).  A warp ran
    // as long as its slowest star (22 of 32 lanes busy, now 30): orbit stage of 10^6,
    // 64 x 10^5, 10^7 stars 148.5, 851, 1246 us, FP64 mode at 10^7 2294; with the
    // rounds from the first, second, third, fourth trial on 149.5, 841, 1230, 2277;
    // 147.5, 837, 1223, 2265; 145.4, 827, 1211, 2253; 146.5, 832, 1217, 2270.
    const bool result = pend;
    __shared__ uint8_t s_owner[256];
    uint8_t* owner = s_owner + (threadIdx.x & ~31u);
    const bool one = __match_any_sync(0xFFFFFFFFu, c) == 0xFFFFFFFFu;
    const Grid GD = grid_of(BA, c < 0 ? 0 : c);
    const uint32_t stp = *step_p;
    for (;;) {
      const unsigned lm = __ballot_sync(0xFFFFFFFFu, live);
      if (!lm) break;
      const int k = __popc(lm), rank = __popc(lm & ((1u << lane) - 1u));
      // 2^lg lanes a star: the largest with k 2^lg <= 32
      const int lg = one ? __clz(2 * k - 1) - 26 : 0;
      const int G = 1 << lg;
      float e = E32, jj = J32, a0 = c0f, a1 = c1f, ff = F32;
      uint32_t iv = idv;
      int mine = t, from = lane;
      bool go = live;
      if (G > 1) {
        if (live) owner[rank] = (uint8_t)lane;
        __syncwarp();
        const int slot = lane >> lg;
        go = slot < k;
        from = go ? owner[slot] : lane;
        __syncwarp();
        e = __shfl_sync(0xFFFFFFFFu, E32, from);
        jj = __shfl_sync(0xFFFFFFFFu, J32, from);
        a0 = __shfl_sync(0xFFFFFFFFu, c0f, from);
        a1 = __shfl_sync(0xFFFFFFFFu, c1f, from);
        ff = __shfl_sync(0xFFFFFFFFu, F32, from);
        iv = __shfl_sync(0xFFFFFFFFu, idv, from);
        mine = __shfl_sync(0xFFFFFFFFu, t, from) + (lane & (G - 1));
      }
      int d = 0;
      unsigned long long over = 0;
      if (go && mine < max_trials) {
        Draws<false> g = draws_of<false>(S, c, iv, stp);
        const U4 w = g.block(kTagRej, (uint32_t)mine);
        d = accept32<kExact>(GD, e, jj, a0, a1, ff, 2.0f * u01f(w.y) - 1.0f, u01f(w.w), over);
      }
      const unsigned acc = __ballot_sync(0xFFFFFFFFu, d > 0);
      const unsigned any = acc | __ballot_sync(0xFFFFFFFFu, d < 0);
      if (G == 1) {
        viol += over;
        if (live) {
          if (d != 0) {
            st = d > 0 ? kSmpAccepted : kSmpPending;
            live = false;
          } else if (++t >= max_trials) {
            live = false;
          }
        }
      } else {
        const unsigned gm = G == 32 ? 0xFFFFFFFFu : (1u << G) - 1u;
        // the executing lanes' group, then the owners'
        const unsigned mg = (any >> (lane & ~(G - 1))) & gm;
        if (go && (!mg || (lane & (G - 1)) <= __ffs(mg) - 1)) viol += over;
        if (live) {
          const unsigned og = (any >> (rank * G)) & gm;
          if (og) {
            const int last = __ffs(og) - 1;
            st = (acc >> (rank * G + last)) & 1u ? kSmpAccepted : kSmpPending;
            t += last;
            live = false;
          } else {
            t += G;
            if (t >= max_trials) {
              t = max_trials;
              live = false;
            }
          }
        }
      }
    }
    pend = false;
    if (result) {
      keys[p] = ((uint64_t)__float_as_uint(F32) << 32) | ((uint64_t)st << 30) |
                (uint64_t)(t & 0x3FFFFFFF);
      pend = st == kSmpPending;
    }
  }
  // pending stars onto the list of k_pending64 (one atomic per warp)
  const unsigned pm = __ballot_sync(__activemask(), pend);
  if (pm) {
    uint32_t base = 0;
    if (lane == __ffs(pm) - 1) base = atomicAdd(pcount, (uint32_t)__popc(pm));
    base = __shfl_sync(__activemask(), base, __ffs(pm) - 1);
    if (pend) plist[base + __popc(pm & ((1u << lane) - 1u))] = (uint32_t)p;
  }
  // violations: one atomic per segment present in the warp
  const unsigned full = __activemask();
  const unsigned peers = __match_any_sync(full, c);
  const unsigned vi = __reduce_add_sync(peers, (unsigned)viol);
  if ((threadIdx.x & 31) == __ffs(peers) - 1 && c >= 0) stat_add(S.stats, c, kStViolations, vi);
}

// Third kernel of the mixed-mode orbit step: every star the FP32 sampler
// left pending (a trial whose accept test FP32 could not decide, mostly
// close to a turning point, where Q vanishes like (1 - |s|)^2) takes that
// trial and the rest of its sequence in FP64; its key slot then holds
// kSmpAccepted and the accepted trial, or kSmpCap.  Most threads find no
// pending star and leave at once.
// one pending star (p = n: an idle lane); counts go to the statistics
// kExact (FP64 mode): F = 1.2 Fx, the points and g as FP64 mode's
template <bool kTaus, bool kExact, bool kAhead>
__device__ __forceinline__ void pending_star(Seg S, int max_trials, const uint32_t* id,
                                             const uint32_t* step_p, BucketArgs BA,
                                             const double4_32a* orb, uint64_t* keys, int64_t p,
                                             int64_t n, const double* Fx, int lanes_each) {
  const int G = kAhead ? lanes_each : 1;
  unsigned long long viol = 0;
  unsigned int n64 = 0;
  int c = -1;
  if (p < n) {
    c = seg_find(S.off, S.n_seg, p);
    const int64_t sb = S.off[c], nbc = S.nb[c], k = p - sb;
    if (k < nbc) {
      const uint64_t res = keys[p];
      const double4_32a o = orb[p];  // E, J, c0, c1 from the turning-point kernel
      Star s;
      s.k = k;
      s.E = o.x;
      s.J = o.y;
      if (lt0(s.E) && ((uint32_t)(res >> 30) & 3u) == kSmpPending) {
        Buckets BK;
        const int4 pr = BA.prm[c];
        BK.start = BA.start + BA.off[c];
        BK.base = BA.base[c];
        BK.shift = pr.x;
        BK.nbk = pr.y;
        BK.lo = pr.z;
        BK.hi = pr.w;
        const double c0 = o.z, c1 = o.w;
        const float c0f = f32_rn(c0), c1f = f32_rn(c1);
        const double F =
            kExact ? 1.2 * Fx[p] : (double)__uint_as_float((uint32_t)(res >> 32));
        uint32_t st = kSmpCap;
        int t = (int)(res & 0x3FFFFFFFull);
        // stream mode: the blocks of trials 0 .. t-1 were the FP32 sampler's
        Draws<kTaus> g = draws_of<kTaus>(S, c, id[p], *step_p);
        g.skip((uint32_t)t);
        // G lanes take G trials at a time; the first accepted one counts, as do
        // the trials up to it
        const int lane = threadIdx.x & 31, sub = lane & (G - 1);
        const unsigned group = (G == 32 ? 0u : 1u << G) - 1u, at = lane - sub;
        for (; t < max_trials; t += G) {
          const int mine = t + sub;
          bool over = false, take = false;
          if (mine < max_trials) {
            const U4 w = g.block(kTagRej, (uint32_t)mine);
            const double sv = sym_double(sym_int(w.x, w.y));
            const int guess =
                shell32_of(BA.node + sb, (int)nbc, BK, c0f, c1f, 2.0f * u01f(w.y) - 1.0f);
            double g64v;
            if (kExact) {
              double rs, ph, Q, L, xq;
              int i;
              point64_div(BA.node + sb, nbc, s, c0, c1, sv, guess, rs, ph, Q, L, xq, i);
              g64v = g_of_point(c1, sv, Q);
            } else {
              double rs, xs, ph, L, Q;
              int i;
              point64(BA.node + sb, nbc, s, c0, c1, sv, guess, rs, xs, ph, L, Q, i);
              g64v = pos_num(Q) ? div_rn((3.0 * c1) * (1.0 - sv * sv), sqrt_rn(Q)) : 0.0;
            }
            over = g64v > F;
            take = F * u01(w.z, w.w) < g64v;
          }
          const unsigned acc = kAhead ? (__ballot_sync(group << at, take) >> at) & group : take;
          const int last = acc ? __ffs(acc) - 1 : G - 1;
          if (mine < max_trials && sub <= last) {
            ++n64;
            viol += over;
          }
          if (acc) {
            st = kSmpAccepted;
            t += last;
            break;
          }
        }
        if (t >= max_trials) t = max_trials;
        if (sub == 0)
          keys[p] = (res & 0xFFFFFFFF00000000ull) | ((uint64_t)st << 30) |
                    (uint64_t)(t & 0x3FFFFFFF);
      }
    }
  }
  const unsigned full = __activemask();
  const unsigned peers = __match_any_sync(full, c);
  const unsigned vi = __reduce_add_sync(peers, (unsigned)viol);
  const unsigned nf = __reduce_add_sync(peers, n64);
  if ((threadIdx.x & 31) == __ffs(peers) - 1 && c >= 0) {
    stat_add(S.stats, c, kStViolations, vi);
    stat_add(S.stats, c, kStFp64Trials, nf);
  }
}

constexpr uint32_t kPendingWarps = 16 * 152;

template <bool kTaus, bool kExact>
__global__ void __launch_bounds__(128) k_pending64(Seg S, int max_trials, const uint32_t* id,
                                                   const uint32_t* step_p, BucketArgs BA,
                                                   const double4_32a* orb, uint64_t* keys,
                                                   const uint32_t* plist,
                                                   const uint32_t* pcount, int64_t n,
                                                   const double* Fx) {
  pdl_enter();
  const uint32_t np = *pcount;
  // A short list goes over more warps, `lanes` stars to each (a warp's walks and
  // trials last as long as its slowest star's), and the lanes left over take
  // trials ahead, which costs no instructions: the orbit stage of 10^3, 10^4 (FP64
  // mode), 10^5, 10^6 stars 42.2, 56.1, 52.7, 165.7 us with one lane a star over four
  // warps per SM, 26.1, 46.3, 37.9, 166.5 with trials ahead, 26.5, 46.3, 35.5, 149.8
  // over sixteen warps per SM (eight: 25.8, 46.3, 35.5, 158.6; 32: 26.4, 45.6, 36.3,
  // 148.7); full warps 44.0, 58.1, 56.0.
  const uint32_t warps = gridDim.x * (blockDim.x / 32), lane = threadIdx.x & 31;
  uint32_t lanes = (np + kPendingWarps - 1) / kPendingWarps;
  lanes = lanes < 32u ? lanes : 32u;
  if (lanes * warps < np) lanes = 32u;
  // ... and the lanes left over take trials ahead
  const int G = kTaus || lanes > 16u ? 1
                : lanes > 8u             ? 2
                : lanes > 4u             ? 4
                : lanes > 2u             ? 8
                : lanes > 1u             ? 16
                                         : 32;
  const uint32_t slot = lane / G;
  for (uint32_t w = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32; w * lanes < np; w += warps) {
    const uint32_t i = w * lanes + slot;
    const int64_t p = slot < lanes && i < np ? (int64_t)plist[i] : n;
    if (!kTaus && G > 1)
      pending_star<kTaus, kExact, true>(S, max_trials, id, step_p, BA, orb, keys, p, n, Fx, G);
    else
      pending_star<kTaus, kExact, false>(S, max_trials, id, step_p, BA, orb, keys, p, n, Fx, 1);
  }
}

// the star's records, and its bin (counted too with cnt) or its sort key
struct BinOut {
  uint32_t* bin = nullptr;
  uint32_t* cnt = nullptr;
  const int64_t* cbase = nullptr;
  const int* esh = nullptr;
};

// s: shell + 1 of a bound star, -1 for an escaped one
__device__ __forceinline__ void put_star(const Seg& S, const BinOut& O, uint64_t* keys, RecA* ra,
                                         RecB* rb, RecA& A, const RecB& B, int64_t p, int c,
                                         int64_t s) {
  if (O.bin) {
    const int64_t nc = S.off[c + 1] - S.off[c];
    if (s < 0) s = nc + 1 + (int64_t)(A.id >> O.esh[c]);
    A.bin = (uint32_t)(O.cbase[c] + s);
    O.bin[p] = A.bin;
    if (O.cnt) {
      // (stars crowding into few bins: the lanes of a bin together, as k_bin_count)
      const unsigned on = __activemask();
      const uint32_t lane = threadIdx.x & 31u, next = __shfl_down_sync(on, A.bin, 1);
      if (__any_sync(on, next == A.bin && lane < 31u)) {
        const unsigned peers = __match_any_sync(on, A.bin);
        if ((int)lane == __ffs(peers) - 1) atomicAdd(O.cnt + A.bin, (uint32_t)__popc(peers));
      } else {
        atomicAdd(O.cnt + A.bin, 1u);
      }
    }
  } else {
    keys[p] = radius_key(A.r, A.id);
  }
  store_rec(ra + p, A);
  store_rec(rb + p, B);
}

// kPrec: 0 FP64 by bisection (Appendix A's kernels: brackets, envelope and
// trials all on the FP64 table), 1 mixed (turning points from
// k_turning_mixed in tp_min, tp_max, FP32 sampler result from k_sample32 /
// k_pending64 in the key slot), 2 FP64 through the mixed kernels (their
// FP64 turning points, FP64 mode's envelope 1.2 Fx (Fx from k_env_eval), the
// accepted point as FP64 mode computes it).  kMinB: resident 256-thread
// blocks to fit (caps registers; 1 = no cap).
template <int kPrec, int kMinB, bool kTaus>
__global__ void __launch_bounds__(256, kMinB) k_orbit(Seg S, int max_trials, const double* r,
                                               const double* x, const double* phi,
                                               const double* vr, const double* vt,
                                               const double* m,
                                               const uint32_t* id, const uint32_t* step_p,
                                               uint64_t* keys, RecA* ra, RecB* rb,
                                               int64_t* esc, OrbitStageOut dbg, BucketArgs BA,
                                               const double* tp_min, const double* tp_max,
                                               const double4_32a* orb,
                                               int64_t n, const double* Rv, double* Rp,
                                               const double* Fx, const double* Av,
                                               double* Ap, BinOut bo, uint32_t* pcount,
                                               unsigned long long* ecount) {
  pdl_enter();
  // the lists' counters, read by the kernels before this one, zero for the next
  // orbit step (two fills less between its kernels)
  if (kPrec != 0 && blockIdx.x == 0 && threadIdx.x == 0) {
    *pcount = 0u;
    if (kPrec == 2) ecount[0] = ecount[1] = 0ull;
  }
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const int c = seg_find(S.off, S.n_seg, p);
  const int64_t sb = S.off[c];
  const int64_t nbc = S.nb[c];
  const int64_t k = p - sb;
  const double rk = r[p];
  const uint32_t idk = id[p];
  const double inf = __longlong_as_double((long long)kInfBits);
  RecA A;
  A.r = rk; A.x = 0.0; A.id = idk; A.bin = 0u;
  RecB B;
  B.c = 0.0; B.w = 0.0;
  // (the star's mass, and its velocities where it keeps them, are read where they
  // are stored: held from here on they spill, and spilled lines leave the L1 under
  // the random node reads, which makes the stage of 10^7 stars 1.35 ms instead of
  // 1.21 in many steps)
  auto keep_velocities = [&]() {
    B.vr = vr[p];
    B.vt = vt[p];
  };
  double x_new = 0.0;
  int shell = -2;  // of r_new in the current table; -2: not found on the way
  double r_new = rk, rmin = rk, rmax = rk, F = 0.0;
  int code = 0, trials = 0;
  unsigned long long viol = 0;
  bool escaped = false;

  if (Rp) Rp[p] = Rv[p];  // the stellar radius goes with the star
  if (Ap) Ap[p] = Av[p];  // and the binary's semi-major axis
  if (k >= nbc) {
    // escaped in an earlier step: stays at the end, ordered by id
    A.m = m[p];
    keep_velocities();
    put_star(S, bo, keys, ra, rb, A, B, p, c, -1);
    if (dbg.code) dbg.code[p] = 1;
    return;
  }
  if (Rv && lt0(Rv[p])) {
    // merged into its partner in this step (sticky spheres): it leaves
    // with no mass, draws nothing, and carries off no energy
    A.r = inf;
    A.m = m[p];
    keep_velocities();
    put_star(S, bo, keys, ra, rb, A, B, p, c, -1);
    if (dbg.code) dbg.code[p] = 1;
    const unsigned full = __activemask();
    const unsigned peers = __match_any_sync(full, c);
    if ((threadIdx.x & 31) == __ffs(peers) - 1)
      atomicAdd((unsigned long long*)(esc + c), (unsigned long long)__popc(peers));
    return;
  }
  const Table64 T{r + sb, x + sb, phi + sb, nbc};
  Star s;
  s.k = k;
  double c0o = 0.0, c1o = 0.0;
  if (kPrec >= 1) {
    // E, J, c0, c1 from the turning-point kernel
    const double4_32a o = orb[p];
    s.E = o.x;
    s.J = o.y;
    c0o = o.z;
    c1o = o.w;
  } else {
    const double vrk = vr[p], vtk = vt[p];
    s.E = T.phi[k] + scale_down<1>(vrk * vrk + vtk * vtk);
    s.J = rk * vtk;
  }
  Draws<kTaus> g = draws_of<kTaus>(S, c, idk, *step_p);
  double ph_new = T.phi[k];

  if (!lt0(s.E)) {
    escaped = true;
    code = 1;
    r_new = inf;
    // energy carried off: the star's energy in the field of the others
    const double vrk = vr[p], vtk = vt[p];
    B.c = T.phi[k] + div_rn(m[p], rk) + scale_down<1>(vrk * vrk + vtk * vtk);
  } else {
    int64_t jmax, jmin;
    Buckets BK;
    if (kPrec >= 1) {
      const int4 pr = BA.prm[c];
      BK.start = BA.start + BA.off[c];
      BK.base = BA.base[c];
      BK.shift = pr.x;
      BK.nbk = pr.y;
      BK.lo = pr.z;
      BK.hi = pr.w;
    }
    if (kPrec == 0) {
      jmax = bisect_rmax64(T, s);
      jmin = bisect_rmin64(T, s);
    } else if (dbg.rmin) {
      // turning points from k_turning_mixed (for the stage outputs)
      rmin = tp_min[p];
      rmax = tp_max[p];
    }
    if (kPrec == 0) {
      rmax = shell_root64(T, s, jmax, true);
      rmin = jmin < 0 ? central_root64(T, s) : shell_root64(T, s, jmin, false);
    }
    const double c0 = kPrec == 0 ? scale_down<1>(rmax + rmin) : c0o;
    const double c1 = kPrec == 0 ? scale_down<2>(rmax - rmin) : c1o;
    if (kPrec == 0) {
      double gmax = 0.0;
      for (int j = 0; j <= 20; ++j) {
        double rs, ph, Q;
        int64_t i;
        double g = g64(T, s, c0, c1, c_s64[j], rs, ph, Q, i);
        if (g > gmax) gmax = g;
      }
      F = 1.2 * gmax;
      if (!(rmax > rmin) || !(F > 0.0)) {
        code = 2;
      } else {
        code = 3;
        double rs_a = 0.0, ph_a = 0.0, Q_a = 0.0;
        for (int t = 0; t < max_trials; ++t) {
          U4 w = g.block(kTagRej, (uint32_t)t);
          const double Xp = u01(w.z, w.w);
          const double sv = sym_double(sym_int(w.x, w.y));  // 2 X - 1, exact
          double rs, ph, Q;
          int64_t i;
          const double g = g64(T, s, c0, c1, sv, rs, ph, Q, i);
          if (g > F) ++viol;
          if (F * Xp < g) {
            rs_a = rs;
            ph_a = ph;
            Q_a = Q;
            shell = (int)i;
            code = 0;
            trials = t + 1;
            break;
          }
        }
        if (code == 3) {
          trials = max_trials;
          draws_keep(S, c, g);
        } else {
          // the accepted point's velocities once the warp's lanes are done
          const double sq = sqrt_rn(Q_a);
          U4 sg = g.block(kTagSgn, 0u);
          draws_keep(S, c, g);
          r_new = rs_a;
          x_new = div_rn(1.0, rs_a);
          B.vr = (sg.x & 1u) ? -sq : sq;
          B.vt = div_rn(s.J, rs_a);
          B.c = T.phi[k] - ph_a;
          ph_new = ph_a;
        }
      }
    } else {
      // the FP32 sampler's result (k_sample32); a pending star continues
      // its trial sequence here in FP64 from the trial near a turning point
      const uint64_t res = keys[p];
      const uint32_t st = (uint32_t)(res >> 30) & 3u;
      int t = (int)(res & 0x3FFFFFFFull);
      F = kPrec == 2 ? 1.2 * Fx[p] : (double)__uint_as_float((uint32_t)(res >> 32));
      if (st == kSmpDegenerate) {
        code = 2;
      } else if (st == kSmpCap) {
        code = 3;
        trials = max_trials;
        g.skip((uint32_t)max_trials);
        draws_keep(S, c, g);
      } else {
        const float c0f = f32_rn(c0), c1f = f32_rn(c1);
        const int nb32 = (int)nbc;
        // (k_pending64 has resolved every pending star to accepted or cap)
        const bool acc = st == kSmpAccepted;
        if (!acc) {
          code = 3;
          trials = max_trials;
          g.skip((uint32_t)max_trials);
          draws_keep(S, c, g);
        } else {
          code = 0;
          trials = t + 1;
          // the accepted point in FP64 from the full 53-bit X, once per
          // star, with the warp's lanes together
          g.skip((uint32_t)t);  // stream mode: the rejected trials' blocks
          const U4 w = g.block(kTagRej, (uint32_t)t);
          const double sv = sym_double(sym_int(w.x, w.y));
          const int guess = shell32_of(BA.node + sb, nb32, BK, c0f, c1f, 2.0f * u01f(w.y) - 1.0f);
          double rs, ph, Q, vtn;
          if (kPrec == 2)  // v_t = J / r
            point64_div(BA.node + sb, nbc, s, c0, c1, sv, guess, rs, ph, Q, vtn, x_new, shell);
          else
            point64(BA.node + sb, nbc, s, c0, c1, sv, guess, rs, x_new, ph, vtn, Q, shell);
          if (!pos_num(Q)) Q = 0.0;
          const double sq = sqrt_rn(Q);
          U4 sg = g.block(kTagSgn, 0u);
          draws_keep(S, c, g);
          r_new = rs;
          B.vr = (sg.x & 1u) ? -sq : sq;
          B.vt = vtn;
          B.c = T.phi[k] - ph;
          ph_new = ph;
        }
      }
    }
  }
  // a star that stays in place has no point from the way: its shell by bisection
  if (!escaped && shell == -2) {
    x_new = T.x[k];
    if (bo.bin) shell = (int)shell_of(T, rk);
  }
  if (code != 0) keep_velocities();
  A.r = r_new;
  A.x = x_new;
  A.m = m[p];
  put_star(S, bo, keys, ra, rb, A, B, p, c, escaped ? -1 : shell + 1);

  // statistics: one atomic per counter per segment present in the warp
  const unsigned full = __activemask();
  const unsigned peers = __match_any_sync(full, c);
  const int lane = threadIdx.x & 31;
  const unsigned tr = __reduce_add_sync(peers, (unsigned)trials);
  const unsigned vi = __reduce_add_sync(peers, (unsigned)viol);
  const unsigned es = __reduce_add_sync(peers, escaped ? 1u : 0u);
  const unsigned dg = __reduce_add_sync(peers, code == 2 ? 1u : 0u);
  const unsigned cp = __reduce_add_sync(peers, code == 3 ? 1u : 0u);
  if (lane == __ffs(peers) - 1) {
    stat_add(S.stats, c, kStTrials, tr);
    stat_add(S.stats, c, kStViolations, vi);
    stat_add(S.stats, c, kStDegenerate, dg);
    stat_add(S.stats, c, kStCapHits, cp);
    if (es) atomicAdd((unsigned long long*)(esc + c), (unsigned long long)es);
  }
  if (dbg.phi_new) dbg.phi_new[p] = ph_new;
  if (dbg.rmin) dbg.rmin[p] = rmin;
  if (dbg.rmax) dbg.rmax[p] = rmax;
  if (dbg.F) dbg.F[p] = F;
  if (dbg.code) dbg.code[p] = code;
  if (dbg.trials) dbg.trials[p] = trials;
}

// ------------------------------------------------------ potential grid
// Grid cells per segment: twice the stars, between 512 and 2^15.
int64_t grid_capacity(int64_t nc) {
  int64_t g = 2 * nc;
  if (g < 512) g = 512;  // p = 0 (a cell per binade) always fits
  if (g > (1 << 15)) g = 1 << 15;
  return g;
}

// per segment: the key range of 1/r over the bound stars, the finest 2^p
// cells per binade (p <= 10) that fit the capacity, Phi_0 and the bound
// mass (Phi = Phi_0 inside the first star; outside the last one Phi falls
// by M_bound per unit of 1/r)
__global__ void k_grid_params(Seg S, const int64_t* esc, bool sub, const double* x,
                              const double* phi, const double4_32a* node, const int64_t* goff,
                              int4* gprm, float4* gaux) {
  pdl_enter();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= S.n_seg) return;
  int64_t nb = S.nb[c];
  if (sub) nb -= esc[c];
  if (nb <= 0) { gprm[c] = make_int4(0, 0, 0, 0); gaux[c] = make_float4(0.f, 0.f, 0.f, 0.f); return; }
  const int64_t sb = S.off[c];
  const uint32_t klo = __float_as_uint((float)x[sb + nb - 1]);
  const uint32_t khi = __float_as_uint((float)x[sb]);
  const int64_t cap = goff[c + 1] - goff[c];
  int p = 10;
  while (p > 0 && (int64_t)((khi >> (23 - p)) - (klo >> (23 - p))) + 2 > cap) --p;
  const int sh = 23 - p;
  const uint32_t key0 = (klo >> sh) << sh;
  const int cells = (int)((khi - key0) >> sh) + 2;
  gprm[c] = make_int4((int)key0, sh, cells < cap ? cells : (int)cap, (int)khi);
  gaux[c] = make_float4((float)phi[sb], (float)node[sb + nb - 1].w, __uint_as_float(key0), 0.f);
}

// The shell of every grid key, largest i with 1/r_i >= key (-1 when none),
// written by the stars (grid_shells_of) in one pass over stars and cells.
__global__ void k_grid_shells(Seg S, const int64_t* esc, bool sub, const double* x,
                              BucketArgs B, int* gshell, int64_t n) {
  pdl_enter();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned mask = __ballot_sync(0xFFFFFFFFu, p < n);
  if (p >= n) return;
  const int c = seg_find(S.off, S.n_seg, p);
  int64_t nb = S.nb[c];
  if (sub) nb -= esc[c];
  const int64_t sb = S.off[c], k = p - sb;
  const int4 pr = B.gprm[c];
  const bool live = k < nb;
  grid_shells_of(mask, live, (int)k, (int)nb, live ? grid_last_cell(x[p], pr) : -1,
                 live && k + 1 < nb ? grid_last_cell(x[p + 1], pr) : -1, pr,
                 gshell + B.goff[c]);
  if (live && k == 0) grid_close(grid_last_cell(x[p], pr), pr, gshell + B.goff[c], 0, 1);
}

__global__ void k_grid_build(Seg S, const int64_t* esc, GridBuild G) {
  pdl_enter();
  grid_build(S, esc, G, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

// per segment: the indexed node range lo..hi, base = bits(x_lo), the
// smallest shift that fits the key range into the segment's capacity, and
// the bucket count
__global__ void k_bucket_params(Seg S, const int64_t* esc, bool sub, const float2* t32,
                                BucketArgs B, uint32_t* base, int4* prm) {
  pdl_enter();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= S.n_seg) return;
  int64_t nb = S.nb[c];
  if (sub) nb -= esc[c];
  if (nb <= 0) { base[c] = 0; prm[c] = make_int4(0, 0, 0, -1); return; }
  const int64_t sb = S.off[c];
  const int tail = nb >= 4096 ? (int)(nb >> 10) : 0;
  const int lo = tail, hi = (int)nb - 1 - tail;
  const uint32_t b0 = __float_as_uint(t32[sb + lo].x);
  const uint32_t b1 = __float_as_uint(t32[sb + hi].x);
  const uint32_t span = b0 >= b1 ? b0 - b1 : 0u;
  const int64_t cap = B.off[c + 1] - B.off[c] - 1;  // buckets that fit
  int sh = 0;
  while ((int64_t)(span >> sh) + 1 > cap) ++sh;
  base[c] = b0;
  prm[c] = make_int4(sh, (int)((span >> sh) + 1), lo, hi);
}

// one thread per indexed star: it writes start[b] for the buckets between
// its predecessor's bucket and its own; the last one closes the table
__global__ void k_bucket_build(Seg S, const int64_t* esc, bool sub, const float2* t32,
                               BucketArgs B, int* start, int64_t n) {
  pdl_enter();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned mask = __ballot_sync(0xFFFFFFFFu, p < n);
  if (p >= n) return;
  const int c = seg_find(S.off, S.n_seg, p);
  int64_t nb = S.nb[c];
  if (sub) nb -= esc[c];
  const int64_t k = p - S.off[c];
  bucket_starts_of(mask, k < nb, (int)k, B.prm[c], B.base[c], __float_as_uint(t32[p].x),
                   k > 0 ? __float_as_uint(t32[p - 1].x) : 0u, start + B.off[c],
                   B.off[c + 1] - B.off[c]);
  if (k == B.prm[c].w)
    bucket_close((int)nb, B.prm[c], B.base[c], __float_as_uint(t32[p].x), start + B.off[c],
                 B.off[c + 1] - B.off[c], 0, 1);
}

// slope of Phi in 1/r across each shell of one table, for callers that
// have the potential but not the masses: (Phi_{k+1} - Phi_k)/(x_k - x_{k+1}),
// with Phi = 0 at 1/r = 0 beyond the last node
__global__ void k_slopes(int64_t n, const double* x, const double* phi, double* M) {
  pdl_enter();
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const double xj = x[k], pj = phi[k];
  const double xj1 = k + 1 < n ? x[k + 1] : 0.0, pj1 = k + 1 < n ? phi[k + 1] : 0.0;
  M[k] = div_rn(pj1 - pj, xj - xj1);
}

}  // namespace

void launch_slopes(int64_t n, const double* x, const double* phi, double* Menc,
                   cudaStream_t st) {
  if (n > 0) launch_k(k_slopes, (unsigned)((n + 255) / 256), 256, 0, st, n, x, phi, Menc);
}

cudaError_t alloc_buckets(BucketWork& B, const SegLayout& L, cudaStream_t st) {
  std::vector<int64_t> off(L.n_seg + 1, 0), goff(L.n_seg + 1, 0);
  for (int c = 0; c < L.n_seg; ++c) {
    const int64_t nc = L.h_off[c + 1] - L.h_off[c];
    // a bucket per star on average over the key range.  With half as many the walks
    // at the ends of a bucket are longer (turning points of 10^6 stars 124 us
    // against 109, of 64 x 10^5 stars 616 against 599; the fill costs 7 and 2 us
    // less); with twice as many the table no longer stays in the L2 (the orbit
    // stage of 10^7 stars 1354 us against 1242).
    off[c + 1] = off[c] + nc + 2;
    goff[c + 1] = goff[c] + grid_capacity(nc);
  }
  B.gcells = goff[L.n_seg];
  const size_t seg = (size_t)L.n_seg;
  Carve C;
  C.put(B.off, off.data(), seg + 1);
  C.put(B.goff, goff.data(), seg + 1);
  C.add(B.start, (size_t)off[seg]);
  C.add(B.base, seg);
  C.add(B.prm, seg);
  C.add(B.gphi, (size_t)B.gcells);
  C.add(B.gshell, (size_t)B.gcells);
  C.add(B.gprm, seg);
  C.add(B.gaux, seg);
  C.add(B.node, (size_t)L.n);
  return C.alloc(B.block, st);
}

void free_buckets(BucketWork& B, cudaStream_t st) {
  if (B.block) cudaFreeAsync(B.block, st);
  B = BucketWork();
}

// fused: also the slopes at the tile seams
static GridBuild grid_args(const SegLayout& L, const double* x, const double* phi, bool nb_sub,
                           bool fused, const BucketWork& B) {
  GridBuild G;
  G.x = x;
  G.phi = phi;
  G.B = B.args();
  G.gshell = B.gshell;
  G.gphi = B.gphi;
  G.gaux = B.gaux;
  G.total = B.gcells;
  G.sub = nb_sub;
  G.fused = fused;
  G.node = B.node;
  G.n_tiles = fused ? L.n_tiles : 0;
  return G;
}

static void launch_grid_build(const SegLayout& L, const GridBuild& G, cudaStream_t st) {
  launch_k(k_grid_build, (unsigned)((G.total + G.n_tiles + 255) / 256), 256, 0, st, L.dev(),
           L.esc_step, G);
}

void launch_grid(const SegLayout& L, const double* x, const double* phi, bool nb_sub,
                 BucketWork& B, cudaStream_t st) {
  if (!L.n || !B.gcells) return;
  launch_k(k_grid_params, (unsigned)((L.n_seg + 127) / 128), 128, 0, st, L.dev(), L.esc_step,
           nb_sub, x, phi, B.node, B.goff, B.gprm, B.gaux);
  launch_k(k_grid_shells, (unsigned)((L.n + 255) / 256), 256, 0, st, L.dev(), L.esc_step, nb_sub, x,
           B.args(), B.gshell, L.n);
  launch_grid_build(L, grid_args(L, x, phi, nb_sub, false, B), st);
}

void launch_potential_tables(const SegLayout& L, const double* r, const double* x,
                             const double* m, double* tile_m, double* tile_mx, double* phi,
                             bool nb_sub, bool sums_ready, BucketWork& B, cudaStream_t st,
                             GridBuild* later, double* recip) {
  if (!L.n) return;
  TableOut T;
  T.start = B.start;
  T.boff = B.off;
  T.base = B.base;
  T.prm = B.prm;
  T.gshell = B.gshell;
  T.goff = B.goff;
  T.gprm = B.gprm;
  T.gaux = B.gaux;
  launch_potential(L, r, x, m, tile_m, tile_mx, phi, nullptr, nb_sub, st, sums_ready, B.node, &T,
                   recip);
  const GridBuild G = grid_args(L, x, phi, nb_sub, true, B);
  if (later) *later = G;
  else launch_grid_build(L, G, st);
}

void launch_buckets(const SegLayout& L, const float2* t32, bool nb_sub, BucketWork& B,
                    cudaStream_t st) {
  if (!L.n) return;
  launch_k(k_bucket_params, (unsigned)((L.n_seg + 127) / 128), 128, 0, st,
      L.dev(), L.esc_step, nb_sub, t32, B.args(), B.base, B.prm);
  launch_k(k_bucket_build, (unsigned)((L.n + 255) / 256), 256, 0, st, L.dev(), L.esc_step, nb_sub,
                                                               t32, B.args(), B.start, L.n);
}

cudaError_t alloc_env(EnvWork& W, int64_t n, cudaStream_t st) {
  const int64_t m = n > 0 ? n : 1;
  W.cap = 2 * m + 1024;  // the pairs: 1.1 per star measured on Plummer models
  Carve C;
  C.zero(W.cnt, 2);
  C.add(W.gmax, (size_t)m);
  C.add(W.star, (size_t)m);
  C.add(W.list, (size_t)W.cap);
  C.add(W.spill, (size_t)m);
  cudaError_t e = C.alloc(W.block, st);
  if (!e) {
    launch_k(k_env_tables, 1, 32, 0, st);
    e = cudaGetLastError();
  }
  return e;
}

void free_env(EnvWork& W, cudaStream_t st) {
  if (W.block) cudaFreeAsync(W.block, st);
  W = EnvWork();
}

void launch_turning(const SegLayout& L, const double* r, const double* x, const double* phi,
                    const double* vr, const double* vt,
                    const BucketArgs& ba, double* tp_min, double* tp_max, double4_32a* orb,
                    int block, cudaStream_t st) {
  if (!L.n) return;
  if (block <= 0) block = 64;
  const unsigned grid = (unsigned)((L.n + block - 1) / block);
  launch_k(k_turning_mixed<5>, grid, block, 0, st, L.dev(), r, x, phi, vr, vt, ba, tp_min,
                                             tp_max, orb, L.n);
}

void launch_orbit(const SegLayout& L, int precision, int max_trials, const double* r,
                  const double* x, const double* phi,
                  const double* vr, const double* vt, const double* m, const uint32_t* id,
                  const uint32_t* step,
                  uint64_t* keys, RecA* ra, RecB* rb, const OrbitStageOut* dbg, int block,
                  int variant, const BucketArgs& ba, double* tp_min, double* tp_max,
                  uint32_t* plist, uint32_t* pcount, cudaStream_t st, bool with_turning,
                  const double* Rv, double* Rp, const EnvWork* env, const double* Av,
                  double* Ap, double4_32a* orb, const BinWork* bins, uint32_t* bin, bool count) {
  if (!L.n) return;
  OrbitStageOut d;
  BinOut bo;
  if (bins) {
    bo.bin = bin;
    bo.cnt = count ? bins->cnt : nullptr;
    bo.cbase = bins->cbase;
    bo.esh = bins->esh;
  }
  EnvWork W;
  if (env) W = *env;
  double* Fx = W.gmax;
  // the envelope's pairs, about 1.1 per star: one thread each (a grid for
  // 1.25 per star, striding over any more)
  const unsigned egrid = (unsigned)((L.n + L.n / 4 + kEnvThreads - 1) / kEnvThreads);
  if (dbg) d = *dbg;
  if (block <= 0) block = 64;
  const unsigned grid = (unsigned)((L.n + block - 1) / block);
  // the pending list is short: a grid of a few blocks per SM walks it
  const unsigned pgrid = (unsigned)((L.n + 31) / 32 < 1216 ? (L.n + 31) / 32 : 1216);
  // precision 0: FP64 through the mixed kernels (kPrec 2); 1 mixed; 2 FP64
  // by bisection (kPrec 0)
  const bool exact = precision == 0;
#define CMC_TURN(B)                                                                          \
  launch_k(k_turning_mixed<5>, grid, block, 0, st, L.dev(), r, x, phi, vr, vt, ba,      \
                                             tp_min, tp_max, orb, L.n)
#define CMC_ORBIT(P, B, T)                                                                  \
  launch_k(k_orbit<P, B, T>, grid, block, 0, st, L.dev(), max_trials, r, x, phi, vr, vt, \
           m, id, step, keys, ra, rb, L.esc_step, d, ba, tp_min, tp_max, orb, L.n, Rv, Rp, Fx, \
           Av, Ap, bo, pcount, W.cnt)
#define CMC_SAMPLED(B, T, X)                                                                \
  do {                                                                                      \
    if (with_turning) CMC_TURN(B);                                                          \
    if (X) {                                                                                \
      const int g = star_lanes(L);                                                          \
      launch_k(g == 8   ? k_env_screen<8>                                                   \
               : g == 4 ? k_env_screen<4>                                                   \
                        : k_env_screen<1>,                                                  \
               (unsigned)((L.n * g + kEnvThreads - 1) / kEnvThreads), kEnvThreads, 0, st,   \
               L.dev(), ba, orb, W, L.n);                                                   \
      launch_k(k_env_eval, egrid, kEnvThreads, 0, st, L.dev(), ba, W);                             \
    }                                                                                       \
    const int ahead = sampler_lanes(L);                                                     \
    launch_k(ahead == 8   ? k_sample32<4, false, X, 8>                                      \
             : ahead == 4 ? k_sample32<4, false, X, 4>                                      \
                          : k_sample32<B, T, X, 1>,                                         \
             ahead > 1 ? (unsigned)((L.n * ahead + 127) / 128) : grid,                      \
             ahead > 1 ? 128 : block, 0, st, L.dev(), max_trials, id, step, ba, orb, keys,  \
             plist, pcount, L.n, Fx);                                                       \
    launch_k(k_pending64<T, X>, pgrid, 128, 0, st, L.dev(), max_trials, id, step, ba, orb, keys,  \
                                             plist, pcount, L.n, Fx);                       \
    CMC_ORBIT(X ? 2 : 1, 5, T);                                                             \
  } while (0)
#define CMC_VARIANTS(X)                                                                     \
  do {                                                                                      \
    if (variant == 1) CMC_SAMPLED(2, false, X);                                             \
    else if (variant == 2) CMC_SAMPLED(3, false, X);                                        \
    else if (variant == 3) CMC_SAMPLED(4, false, X);                                        \
    else if (variant == 4) CMC_SAMPLED(5, false, X);                                        \
    else if (variant == 5) CMC_SAMPLED(6, false, X);                                        \
    else if (variant == 6) CMC_SAMPLED(8, false, X);                                        \
    else CMC_SAMPLED(1, false, X);                                                          \
  } while (0)
  if (precision == 2) {
    if (L.taus) CMC_ORBIT(0, 1, true);
    else CMC_ORBIT(0, 1, false);
  } else if (L.taus) {
    // stream mode: one launch shape of the sampler
    if (exact) CMC_SAMPLED(5, true, true);
    else CMC_SAMPLED(5, true, false);
  } else if (exact) {
    CMC_VARIANTS(true);
  } else {
    CMC_VARIANTS(false);
  }
#undef CMC_VARIANTS
#undef CMC_SAMPLED
#undef CMC_TURN
#undef CMC_ORBIT
}

CMC_DEBUG_SITE_ACCESSOR

}  // namespace cmc
