// Relaxation timestep (Eq. 7 on fixed bins of consecutive stars, section
// 3.3) and two-body relaxation between radial neighbours (section 2.1 step
// 3(i)).  Both are FP64 and evaluate, operation for operation, the same
// expressions as the independent FP64 statement of the method.
#include "cmc_host.hpp"

namespace cmc {

namespace {

// The timesteps over the innermost P = min(300, nb) bound stars of each
// segment (summed in star order, as the FP64 statement of the method does),
// into the segment's timestep (the minimum with Eq. 7's).  With stellar radii R,
// Eq. 8's collision timestep
//   1 / T_coll = 16 sqrt(pi) n_s <R^2> sigma (1 + G <M R> / (2 sigma^2 <R^2>)),
// n_s = 3 (P - 1) / (4 pi (r_{P-1}^3 - r_0^3)), sigma^2 = <v_r^2 + v_t^2> / 3.
// With binaries (semi-major axes A > 0, the star's mass the binary's),
// Eqs. 9 and 10:
//   1 / T_bb = 16 sqrt(pi) n_b X_bb^2 <a^2> sigma (1 + G <M a> / (2 sigma^2 X_bb <a^2>))
//   1 / T_bs = 4 sqrt(pi) n_s X_bs^2 <a^2> sigma (1 + G <M> <a> / (sigma^2 X_bs <a^2>))
// with n_b, n_s the central density times the binaries' and singles' shares
// of the P stars, <a^2>, <M a>, <a> over the binaries, <M> over all P.
// One block of k_bins per segment: its threads take the stars' terms, the seven
// sums run side by side in seven lanes of a warp (a chain of P additions in star
// order; a term that does not count is a 0 and leaves the sum as it is).  Bound
// by that chain and the formulas after it; a thread per segment that took the
// terms too, in a kernel of its own, took 200 us; this
// takes 13 more than the bins alone.
struct Central {
  const double *R = nullptr, *A = nullptr;
  double x_bb = 0.0, x_bs = 0.0;
};
constexpr int kCentralStars = 300;
enum { kCenV, kCenR, kCenMR, kCenM, kCenA, kCenA2, kCenMA, kCenSums };

__device__ __forceinline__ void central_timestep(const Seg& S, int c, const double* r,
                                                 const double* vr, const double* vt,
                                                 const double* m, const Central& C) {
  __shared__ double s_t[kCenSums][kCentralStars + 1];
  const int64_t nb = S.nb[c], sb = S.off[c];
  const int P = nb < kCentralStars ? (int)nb : kCentralStars;
  if (P < 2) return;  // (one segment a block: all its threads)
  int nbin = 0;
  for (int k0 = 0; k0 < P; k0 += blockDim.x) {
    const int k = k0 + threadIdx.x;
    bool binary = false;
    if (k < P) {
      const int64_t p = sb + k;
      const double mk = m[p], Rk = C.R ? C.R[p] : 0.0, Ak = C.A ? C.A[p] : 0.0;
      binary = Ak > 0.0;
      s_t[kCenV][k] = vr[p] * vr[p] + vt[p] * vt[p];
      s_t[kCenR][k] = Rk * Rk;
      s_t[kCenMR][k] = mk * Rk;
      s_t[kCenM][k] = mk;
      s_t[kCenA][k] = binary ? Ak : 0.0;
      s_t[kCenA2][k] = binary ? Ak * Ak : 0.0;
      s_t[kCenMA][k] = binary ? mk * Ak : 0.0;
    }
    nbin += __syncthreads_count(binary);
  }
  if (threadIdx.x >= 32) return;
  const int lane = threadIdx.x;
  double sum = 0.0;
  if (lane < kCenSums) {
#pragma unroll 10
    for (int k = 0; k < P; ++k) sum = sum + s_t[lane][k];
  }
  auto total = [&](int l) { return __shfl_sync(0xFFFFFFFFu, sum, l); };
  const double sv = total(kCenV), sr = total(kCenR), smr = total(kCenMR), sm = total(kCenM),
               sa = total(kCenA), sa2 = total(kCenA2), sma = total(kCenMA);
  if (lane != 0) return;
  const double* rr = r + sb;
  const double vol = rr[P - 1] * rr[P - 1] * rr[P - 1] - rr[0] * rr[0] * rr[0];
  if (!(vol > 0.0)) return;
  const double ns = (3.0 * (double)(P - 1)) / ((4.0 * kPi) * vol);
  const double inf = __longlong_as_double(0x7FF0000000000000ll);
  const double sig2 = (sv / (double)P) / 3.0;
  const double sig = sig2 > 0.0 ? sqrt(sig2) : 0.0;
  double Tmin = inf;
  if (C.R) {
    const double R2 = sr / (double)P;
    const double MR = smr / (double)P;
    if (R2 > 0.0 && sig2 > 0.0) {
      double inv = (((16.0 * sqrt(kPi)) * ns) * R2) * sig;
      inv = inv * (1.0 + MR / ((2.0 * sig2) * R2));
      const double T = 1.0 / inv;
      if (T < Tmin) Tmin = T;
    }
  }
  if (C.A && nbin > 0 && sig2 > 0.0) {
    const double a2 = sa2 / (double)nbin, ma = sma / (double)nbin, am = sa / (double)nbin;
    const double mm = sm / (double)P;
    const double nbd = ns * ((double)nbin / (double)P);
    const double nsd = ns * ((double)(P - nbin) / (double)P);
    if (nbin < P) {
      double inv = (((4.0 * sqrt(kPi)) * nsd) * ((C.x_bs * C.x_bs) * a2)) * sig;
      inv = inv * (1.0 + (mm * am) / ((sig2 * C.x_bs) * a2));
      const double T = 1.0 / inv;
      if (T < Tmin) Tmin = T;
    }
    double inv = (((16.0 * sqrt(kPi)) * nbd) * ((C.x_bb * C.x_bb) * a2)) * sig;
    inv = inv * (1.0 + ma / (((2.0 * sig2) * C.x_bb) * a2));
    const double T = 1.0 / inv;
    if (T < Tmin) Tmin = T;
  }
  if (Tmin < inf)
    atomicMin((unsigned long long*)(S.dt_bits + c), (unsigned long long)__double_as_longlong(Tmin));
}

// Bin b of a segment covers sorted positions [b*bs, min((b+1)*bs, nb)).  For P
// >= 2 stars:
//   n = 3 (P-1) / (4 pi (r_last^3 - r_first^3))
//   <v_rel> = mean over pairs (2j, 2j+1) of sqrt(v1^2 + v2^2)
//   <(M1+M2)^2> = mean over the same pairs of (m1 + m2)^2
//   T_b = pref <v_rel>^3 / (lnL n <(M1+M2)^2>),  pref = (theta_max/(pi/2)) (pi/32)
// and the segment's timestep is the minimum of T_b.
// kPairs: a thread per pair takes the pair's two terms (whole bins of a block at a
// time), then a thread per bin sums them in star order and finishes the bin, so
// that a bin's chain of dependent operations is its additions and not its roots;
// else a thread per bin does all of it.  The chain and the loads' latency bound
// few bins, the FP64 pipe many (there the pairs' threads wait at the barriers for
// the bins'): 10.5 us by pairs, 18.4 by bins at 10^5 stars, 13.8 and 18.5 at 4 x
// 10^5, 19.9 and 20.1 at 7 x 10^5 (35,000 bins: the line), 26.6 and 25.0 at 10^6,
// 177 and 128 at 10^7.
// kCentral: the first n_seg blocks take the central timesteps.
constexpr int64_t kBinsByPairs = 32768;
constexpr int kBinThreads = 256;

// a block's bins, and of each bin's `all` pairs those taken at a time
struct BinShape {
  int all, pairs, bins;
};
__host__ __device__ __forceinline__ BinShape bin_shape(int bs, bool by_pairs) {
  BinShape w;
  w.all = bs / 2;
  w.pairs = w.all < kBinThreads ? w.all : kBinThreads;
  w.bins = by_pairs ? kBinThreads / w.pairs : kBinThreads;
  return w;
}

template <bool kCentral, bool kPairs>
__global__ void __launch_bounds__(kBinThreads, kCentral ? 5 : 6) k_bins(
    Seg S, int bs, double pref, const double* r, const double* vr, const double* vt,
    const double* m, double* nbin, Central C) {
  pdl_enter();
  int64_t blk = blockIdx.x;
  if (kCentral) {
    if (blk < S.n_seg) {
      central_timestep(S, (int)blk, r, vr, vt, m, C);
      return;
    }
    blk -= S.n_seg;
  }
  __shared__ unsigned long long s_min[kBinThreads / 32];
  __shared__ int s_seg0;
  const int t = threadIdx.x;
  const BinShape W = bin_shape(bs, kPairs);
  const int G = W.bins;
  const int64_t n_bins = S.bin_off[S.n_seg], b0 = blk * G;
  if (t == 0) s_seg0 = seg_find(S.bin_off, S.n_seg, b0);
  // bin b: its segment, number there, first star and stars
  auto bin_of = [&](int64_t b, int& c, int64_t& lb, int64_t& first, int64_t& P) {
    c = seg_find(S.bin_off, S.n_seg, b);
    lb = b - S.bin_off[c];
    const int64_t nbc = S.nb[c];
    first = lb * bs;
    P = first < nbc ? (nbc - first < bs ? nbc - first : bs) : 0;
    first += S.off[c];
  };
  // a pair's terms
  auto pair = [&](int64_t a, double& v, double& mm) {
    // (two of the five products on the integer pipes: the kernel is bound by
    // the FP64 pipe)
    const double va2 = mul_rn(vr[a], vr[a]) + vt[a] * vt[a];
    const double vb2 = mul_rn(vr[a + 1], vr[a + 1]) + vt[a + 1] * vt[a + 1];
    const double ms = m[a] + m[a + 1];
    v = sqrt_rn(va2 + vb2);
    mm = ms * ms;
  };
  double sv = 0.0, sm = 0.0;
  if (kPairs) {
    __shared__ double s_v[3 * kBinThreads / 2], s_m[3 * kBinThreads / 2];
    const int H = W.pairs, pitch = H | 1;  // G pitch <= G (H + 1) <= 3/2 kBinThreads
    const int g = t / H, j = t - g * H;    // pair j (of every H) of bin b0 + g
    int64_t ga = 0;
    int q = 0;  // the bin's pairs
    if (g < G && b0 + g < n_bins) {
      int c;
      int64_t lb, P;
      bin_of(b0 + g, c, lb, ga, P);
      q = (int)(P / 2);
    }
    for (int j0 = 0; j0 < W.all; j0 += H) {
      if (g < G) {
        double v = 0.0, mm = 0.0;  // (leaves the sums as they are)
        if (j0 + j < q) pair(ga + 2 * (int64_t)(j0 + j), v, mm);
        s_v[g * pitch + j] = v;
        s_m[g * pitch + j] = mm;
      }
      __syncthreads();
      if (t < G) {
        for (int i = 0; i < H; ++i) {
          sv = sv + s_v[t * pitch + i];
          sm = sm + s_m[t * pitch + i];
        }
      }
      __syncthreads();
    }
  } else {
    __syncthreads();  // s_seg0
    if (b0 + t < n_bins) {
      int c;
      int64_t lb, first, P;
      bin_of(b0 + t, c, lb, first, P);
      for (int64_t j = 0; j < P / 2; ++j) {
        double v, mm;
        pair(first + 2 * j, v, mm);
        sv = sv + v;
        sm = sm + mm;
      }
    }
  }
  const int64_t b = b0 + t;
  unsigned long long tb = 0x7FF0000000000000ull;  // +inf
  int c = s_seg0;
  if (t < G && b < n_bins) {
    int64_t lb, first, P;
    bin_of(b, c, lb, first, P);
    double n = 0.0;
    if (P >= 2) {
      const double rf = r[first], rl = r[first + P - 1];
      const double vol = rl * rl * rl - rf * rf * rf;
      if (vol > 0.0) {
        n = div_rn(3.0 * (double)(P - 1), (4.0 * kPi) * vol);
        const double qd = (double)(P / 2);
        const double v = div_rn(sv, qd);
        const double msq = div_rn(sm, qd);
        const double num = pref * (v * v * v);
        const double den = (S.lnL[c] * n) * msq;
        if (den > 0.0) {
          const double T = div_rn(num, den);
          if (T < __longlong_as_double(0x7FF0000000000000ll))
            tb = (unsigned long long)__double_as_longlong(T);
        }
      }
    }
    nbin[b] = n;
    // an outside bound on the segment's timestep (Eq. 11's stellar-evolution
    // step, say), with its first bin
    if (lb == 0 && S.dt_cap) {
      const double cap = S.dt_cap[c];
      if (cap > 0.0 && cap < __longlong_as_double(0x7FF0000000000000ll)) {
        const unsigned long long cb = (unsigned long long)__double_as_longlong(cap);
        tb = cb < tb ? cb : tb;
      }
    }
  }
  // positive doubles order like their bit patterns: min over the block for
  // the block's first segment, direct atomics for any other segment
  unsigned long long mine = (c == s_seg0) ? tb : 0x7FF0000000000000ull;
  if (c != s_seg0 && tb != 0x7FF0000000000000ull)
    atomicMin((unsigned long long*)(S.dt_bits + c), tb);
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long y = __shfl_down_sync(0xffffffffu, mine, o);
    mine = y < mine ? y : mine;
  }
  if ((t & 31) == 0) s_min[t >> 5] = mine;
  __syncthreads();
  if (t == 0) {
    unsigned long long v = s_min[0];
    for (int w = 1; w < kBinThreads / 32; ++w) v = s_min[w] < v ? s_min[w] : v;
    if (v != 0x7FF0000000000000ull) atomicMin((unsigned long long*)(S.dt_bits + s_seg0), v);
  }
}

// One thread per pair slot: stars a = 2j and b = 2j + 1 of a segment.  The
// pair's random draws come from its first star (counters keyed by its id,
// or its stream, kept after the draws).  kMinB: resident 128-thread blocks
// to fit per SM (caps the registers; 1 = no cap), a launch shape only.
//
// With stellar radii (col.R) the pair may merge instead (sticky spheres,
// section 2.1 step 3(iii)): with probability n pi (R1 + R2)^2 (1 + 2 G
// (m1 + m2) / ((R1 + R2) |w|^2)) |w| dt, decided by one draw of the pair
// after the azimuth psi, star a takes the total mass, the pair's 3-D
// momentum and the radius (R1^3 + R2^3)^(1/3); star b gets mass 0 and
// radius -1 (it leaves in the orbit step).  The merger's change of K + W,
// -(m1 m2 / (m1 + m2)) |w|^2 / 2 + m_b (Phi_a - Phi_b) + m_a m_b / r_a,
// is counted (fixed point, 2^-62).
struct Collide {
  double* R = nullptr;        // stellar radii (null: no collisions)
  const double* r = nullptr;  // the current radii and potential
  const double* phi = nullptr;
};

//
// kTwo (few pairs, counter draws): two lanes a pair.  Each draws one of the two
// angles, takes one of each two roots that do not depend on each other, and
// finishes one of the stars: the stage of 10^3, 10^4, 3 x 10^4 stars 16.3, 17.4, 17.9 us
// with a lane a pair, 14.5, 14.9, 16.9 with two; 22.4 and 28.9 at 10^5, where the
// FP64 pipe has work enough (the rule is relax_two_lanes).

template <bool kTaus, int kMinB, bool kCol, bool kTwo>
__global__ void __launch_bounds__(128, kMinB) k_relax(Seg S, int bs, double* vr, double* vt,
                                               double* m, const uint32_t* id,
                                               const double* nbin, const uint32_t* step_p,
                                               Collide col) {
  pdl_enter();
  const int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / (kTwo ? 2 : 1);
  const bool second = kTwo && (threadIdx.x & 1u);  // the pair's second lane
  const unsigned both = 3u << (threadIdx.x & 30u);
  auto of = [&](int l, double v) {  // lane l's value of the pair's two
    return __shfl_sync(both, v, (int)(threadIdx.x & 30u) + l);
  };
  if (p >= S.pair_off[S.n_seg]) return;
  const int c = seg_find(S.pair_off, S.n_seg, p);
  const int64_t j = p - S.pair_off[c];
  const int64_t la = 2 * j;
  if (la + 1 >= S.nb[c]) return;
  const int64_t a = S.off[c] + la, b = a + 1;
  if (!CMC_IN(S.bin_off[c] + la / bs, S.bin_off[c + 1])) return;
  const double n = nbin[S.bin_off[c] + la / bs];
  const double m1 = m[a], m2 = m[b];
  const double msum = m1 + m2;
  const double dt = __longlong_as_double((long long)S.dt_bits[c]);
  const double lnL = S.lnL[c];
  // no density, no mass, or no positive Coulomb logarithm: no deflection
  if (!pos_num(n) || !pos_num(msum) || !pos_num(lnL) || !lt_inf(dt)) return;
  Draws<kTaus> g = draws_of<kTaus>(S, c, id[a], *step_p);
  int fails = 0;
  double cpsi, spsi, cphi, sphi;
  bool got_phi = true;
  if (kTwo) {
    double ca, sa;
    const bool got = disk_angle(g, second ? kTagPhi : kTagPsi, ca, sa);
    cpsi = of(0, ca), spsi = of(0, sa);
    cphi = of(1, ca), sphi = of(1, sa);
    const unsigned ok = __ballot_sync(both, got) >> (threadIdx.x & 30u);
    if (!(ok & 1u)) ++fails;
    got_phi = (ok >> 1) & 1u;
  } else if (!disk_angle(g, kTagPsi, cpsi, spsi)) {
    ++fails;
  }
  const double v1x = vr[a], v1y = vt[a], v1z = 0.0;
  const double v2x = vr[b], vtb = vt[b];
  const double v2y = mul_rn(vtb, cpsi), v2z = mul_rn(vtb, spsi);
  const double wx = v1x - v2x, wy = v1y - v2y, wz = v1z - v2z;
  const double wyy = mul_rn(wy, wy), wzz = mul_rn(wz, wz);
  const double w2 = (mul_rn(wx, wx) + wyy) + wzz;
  if (!pos_num(w2)) {
    draws_keep(S, c, g);
    if (fails && !second) stat_add(S.stats, c, kStAngleFails, (unsigned long long)fails);
    return;
  }
  const double wp2 = wyy + wzz;
  double w, wp = 0.0;
  if (kTwo) {
    const double q = sqrt_rn_nl(second ? wp2 : w2);
    w = of(0, q), wp = of(1, q);
  } else {
    w = sqrt_rn_nl(w2);
  }
  if (kCol) {
    const double R1 = col.R[a], R2 = col.R[b];
    if (R1 + R2 > 0.0) {
      const double Rs = R1 + R2;
      const double focus = 1.0 + div_rn_nl(2.0 * msum, Rs * w2);
      const double sig = (kPi * (Rs * Rs)) * focus;
      const double Pc = ((sig * n) * w) * dt;
      const U4 cw = g.block(kTagCol, 0u);
      if (u01(cw.x, cw.y) < Pc) {
        const double vcx = div_rn_nl(m1 * v1x + m2 * v2x, msum);
        const double vcy = div_rn_nl(m1 * v1y + m2 * v2y, msum);
        const double vcz = div_rn_nl(m1 * v1z + m2 * v2z, msum);
        const double dW = m2 * (col.phi[a] - col.phi[b]) + div_rn_nl(m1 * m2, col.r[a]);
        const double dK = (0.5 * div_rn_nl(m1 * m2, msum)) * w2;
        draws_keep(S, c, g);
        if (kTwo) __syncwarp(both);  // (both have read the pair)
        if (second) return;
        vr[a] = vcx;
        vt[a] = sqrt_rn_nl(vcy * vcy + vcz * vcz);
        m[a] = m1 + m2;
        col.R[a] = cbrt_newton(R1 * R1 * R1 + R2 * R2 * R2);
        m[b] = 0.0;
        col.R[b] = -1.0;
        stat_add(S.stats, c, kStCollisions, 1ull);
        const long long e = __double2ll_rn((dW - dK) * 4611686018427387904.0);  // 2^62
        stat_add(S.stats, c, kStCollisionEnergy, (unsigned long long)e);
        if (fails) stat_add(S.stats, c, kStAngleFails, (unsigned long long)fails);
        return;
      }
    }
  }
  // sin^2(beta/2) = min(1, 2 pi G^2 (m1+m2)^2 n lnL dt / |w|^3)
  double num = (2.0 * kPi) * msum;
  num = num * msum;
  num = num * n;
  num = num * lnL;
  num = num * dt;
  // e1 = (w x xhat)/|w x xhat| = (0, wz, -wy)/|.| (yhat for radial w);
  // u = w x e1 has length |w| and completes the frame perpendicular to w
  double e1y = 1.0, e1z = 0.0, s2;
  const bool across = pos_num(wp2);
  if (kTwo) {
    const double q = div_rn_nl(second ? wz : num, second ? (across ? wp : 1.0) : w2 * w);
    s2 = of(0, q);
    if (across) e1y = of(1, q);
  } else {
    s2 = div_rn_nl(num, w2 * w);
  }
  if (!le1(s2)) s2 = 1.0;
  // cos(beta) = 1 - 2 sin^2(beta/2), sin(beta) = 2 sin(beta/2) cos(beta/2)
  const double cosb = 1.0 - scale_up<1>(s2);
  double sinb;
  if (kTwo) {
    const double q = sqrt_rn_nl(second ? 1.0 - s2 : s2);
    sinb = scale_up<1>(of(0, q)) * of(1, q);
    if (!got_phi) ++fails;
  } else {
    sinb = scale_up<1>(sqrt_rn_nl(s2)) * sqrt_rn_nl(1.0 - s2);
    if (!disk_angle(g, kTagPhi, cphi, sphi)) ++fails;
  }
  draws_keep(S, c, g);
  if (across) {
    if (!kTwo) {
      wp = sqrt_rn_nl(wp2);
      e1y = div_rn_nl(wz, wp);
    }
    e1z = div_rn_nl(-wy, wp);
  }
  const double ux = wy * e1z - wz * e1y;
  const double uy = -(wx * e1z);
  const double uz = wx * e1y;
  const double a1 = w * cphi;
  // w' = w cos(beta) + sin(beta) (|w| cos(phi) e1 + sin(phi) u)
  const double wpx = wx * cosb + sinb * (sphi * ux);
  const double wpy = wy * cosb + sinb * (a1 * e1y + sphi * uy);
  const double wpz = wz * cosb + sinb * (a1 * e1z + sphi * uz);
  const double dwx = wpx - wx, dwy = wpy - wy, dwz = wpz - wz;
  // The products on the integer pipes (these, the frame's and |w|^2 above, the
  // angles' in disk_angle: 17 of the pair's 44) balance the FP64 pipe's load
  // against the issue slots: 0.757 ms at N = 1e7, 0.853 with only these six
  // there, 0.77 to 0.80 with other groups, 0.95 with all (shared body).
  if (kTwo) {
    const double f = div_rn_nl(second ? m1 : m2, msum);
    const double tx = mul_rn(f, dwx), ty = mul_rn(f, dwy), tz = mul_rn(f, dwz);
    const double px = second ? v2x - tx : v1x + tx, py = second ? v2y - ty : v1y + ty,
                 pz = second ? v2z - tz : v1z + tz;
    const int64_t at = second ? b : a;
    const double pt = sqrt_rn_nl(py * py + pz * pz);
    __syncwarp(both);  // (both have read the pair)
    vr[at] = px;
    vt[at] = pt;
    if (fails && !second) stat_add(S.stats, c, kStAngleFails, (unsigned long long)fails);
    return;
  }
  const double f1 = div_rn_nl(m2, msum), f2 = div_rn_nl(m1, msum);
  const double p1x = v1x + mul_rn(f1, dwx), p1y = v1y + mul_rn(f1, dwy), p1z = v1z + mul_rn(f1, dwz);
  const double p2x = v2x - mul_rn(f2, dwx), p2y = v2y - mul_rn(f2, dwy), p2z = v2z - mul_rn(f2, dwz);
  vr[a] = p1x;
  vt[a] = sqrt_rn_nl(p1y * p1y + p1z * p1z);
  vr[b] = p2x;
  vt[b] = sqrt_rn_nl(p2y * p2y + p2z * p2z);
  if (fails) stat_add(S.stats, c, kStAngleFails, (unsigned long long)fails);
}

// Starting states of the Tausworthe streams: slot e of segment c (id =
// e - base[c]) gets T^(id 2^80) of the segment's seeded words, T^(id 2^80)
// as the product of the matrices P_b = T^(2^(80 + b)) over the bits of id.
// P: [4 components][32 bits b][32 columns], a column = the image of one bit.
__global__ void k_taus_init(int64_t slots, int n_seg, const int64_t* base, const uint4* words,
                            const uint32_t* P, uint4* table) {
  pdl_enter();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= slots) return;
  const int c = seg_find(base, n_seg, e);
  const uint64_t idv = (uint64_t)(e - base[c]);
  const uint4 w = words[c];
  uint32_t v[4] = {w.x, w.y, w.z, w.w};
  for (int j = 0; j < 4; ++j)
    for (int b = 0; b < 32; ++b) {
      if (!((idv >> b) & 1ull)) continue;
      const uint32_t* col = P + ((size_t)j * 32 + b) * 32;
      uint32_t r = 0u;
      for (int i = 0; i < 32; ++i)
        if ((v[j] >> i) & 1u) r ^= col[i];
      v[j] = r;
    }
  table[e] = make_uint4(v[0], v[1], v[2], v[3]);
}

}  // namespace

void launch_taus_init(int64_t slots, int n_seg, const int64_t* base, const uint4* words,
                      const uint32_t* P, uint4* table, cudaStream_t st) {
  if (slots > 0)
    launch_k(k_taus_init, (unsigned)((slots + 255) / 256), 256, 0, st, slots, n_seg, base, words, P,
                                                                 table);
}

void launch_bins(const SegLayout& L, const double* r, const double* vr, const double* vt,
                 const double* m, double* nbin, double pref, cudaStream_t st, const double* R,
                 const double* A, double x_bb, double x_bs) {
  if (!L.n_bins) return;
  const bool pairs = L.n_bins <= kBinsByPairs;
  const int G = bin_shape(L.bin_size, pairs).bins;
  const bool central = R || A;
  Central C;
  C.R = R;
  C.A = A;
  C.x_bb = x_bb;
  C.x_bs = x_bs;
  launch_k(central ? (pairs ? k_bins<true, true> : k_bins<true, false>)
                   : (pairs ? k_bins<false, true> : k_bins<false, false>),
           (unsigned)((L.n_bins + G - 1) / G + (central ? L.n_seg : 0)), kBinThreads, 0, st,
           L.dev(), L.bin_size, pref, r, vr, vt, m, nbin, C);
}

template <int kMinB>
static void relax_shape(const SegLayout& L, double* vr, double* vt, double* m,
                        const uint32_t* id, const double* nbin, const uint32_t* step,
                        const Collide& col, cudaStream_t st) {
  const bool two = relax_two_lanes(L);
  const unsigned grid = (unsigned)((L.n_pairs * (two ? 2 : 1) + 127) / 128);
  // (the collision code only in the kernels that need it: it costs
  // registers)
  const auto kernel = L.taus  ? (col.R ? k_relax<true, kMinB, true, false>
                                       : k_relax<true, kMinB, false, false>)
                      : two   ? (col.R ? k_relax<false, 1, true, true>
                                       : k_relax<false, 1, false, true>)
                              : (col.R ? k_relax<false, kMinB, true, false>
                                       : k_relax<false, kMinB, false, false>);
  launch_k(kernel, grid, 128, 0, st, L.dev(), L.bin_size, vr, vt, m, id, nbin, step, col);
}

void launch_relax(const SegLayout& L, double* vr, double* vt, double* m, const uint32_t* id,
                  const double* nbin, const uint32_t* step, cudaStream_t st, int variant,
                  double* R, const double* r, const double* phi) {
  if (!L.n_pairs) return;
  Collide col;
  col.R = R;
  col.r = r;
  col.phi = phi;
  // variants: registers capped for 1 (no cap), 6 or 8 resident blocks per SM
  if (variant == 1) relax_shape<6>(L, vr, vt, m, id, nbin, step, col, st);
  else if (variant == 2) relax_shape<8>(L, vr, vt, m, id, nbin, step, col, st);
  else relax_shape<1>(L, vr, vt, m, id, nbin, step, col, st);
}


CMC_DEBUG_SITE_ACCESSOR

}  // namespace cmc
