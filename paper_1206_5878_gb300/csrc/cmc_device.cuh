// Device-side building blocks shared by the kernels of the Henon Monte Carlo
// timestep (Pattabiraman et al., section 2.1): counter-based random numbers,
// the segment (cluster) layout, error flags, and the shell potential of
// Eqs. 1 and 6 evaluated from the sorted table.
//
// Every kernel is compiled with --fmad=false: each floating-point operation
// is one IEEE-754 round-to-nearest operation in the order written, so the
// FP64 path reproduces an independent FP64 statement of the same method bit
// for bit.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace cmc {

// ---------------------------------------------------------------- sizes
constexpr int kTile = 4096;          // elements per tile (sort, gather, scans)
constexpr int kBins = 256;           // radix digits per pass (8 bits)
constexpr double kPi = 3.14159265358979323846;

// stream tags (third counter word of the per-star random stream)
constexpr uint32_t kTagPsi = 0;      // relaxation: azimuth of star 2's v_t
constexpr uint32_t kTagPhi = 1;      // relaxation: azimuth of the deflection
constexpr uint32_t kTagRej = 2;      // orbit: rejection trials
constexpr uint32_t kTagSgn = 3;      // orbit: sign of the new v_r
constexpr uint32_t kTagCol = 4;      // relaxation pair: sticky-sphere collision draw

// escaped stars sort after every finite radius, by id: key 0x7FF0...0 | id
// << 20, above every finite radius (the radix sort orders by the top
// 40 bits and puts runs equal in them -- escapers whose ids differ only in
// their low 4 bits -- in (key, id) order, which for these keys is id order)
constexpr uint64_t kEscKeyBase = 0x7FF0000000000000ull;

// Debug builds (-DCMC_DEBUG, libcmc_debug.so): index checks at the table
// probes and scatters that a wrong bracket, bucket or segment offset would
// send out of range.  A failed check records the first failing site of its
// translation unit (CMC_TU x 100000 + source line) in that unit's
// g_debug_site, and the access is skipped; release builds compile the
// checks to nothing.
#ifndef CMC_TU
#define CMC_TU 0
#endif
#ifdef CMC_DEBUG
static __device__ unsigned int g_debug_site = 0u;
__device__ __forceinline__ bool debug_in(unsigned long long i, unsigned long long n,
                                         unsigned site) {
  if (i < n) return true;
  atomicCAS(&g_debug_site, 0u, site);
  return false;
}
#define CMC_IN(i, n) \
  ::cmc::debug_in((unsigned long long)(i), (unsigned long long)(n), CMC_TU * 100000u + __LINE__)
#else
#define CMC_IN(i, n) true
#endif

// error bits (fatal: they poison the context)
enum : uint32_t {
  kErrTimeout = 1u << 0,   // a bounded device wait gave up
  kErrTies = 1u << 1,      // a run of equal radii too long to order by id
  kErrInput = 1u << 2,     // invalid input state
  kErrNonFinite = 1u << 3, // a non-finite velocity appeared
};

// per-segment statistics (64-bit counters)
enum : int {
  kStEscaped = 0, kStDegenerate, kStCapHits, kStTrials, kStViolations,
  kStClamps, kStAngleFails, kStTies, kStFp64Trials, kStClampEnergy, kStCollisions,
  kStCollisionEnergy, kStEnvelope64, kStCount
};
// (slot 15: the collision count at the last step end, to tell this step's
// merged-away stars from its escapers)
constexpr int kStCollisionsSeen = 15;
constexpr int kStStride = 16;        // counters reserved per segment
constexpr int kDiagFields = 10;      // doubles per diagnostics record

// Programmatic dependent launch (launch_k): a kernel of a timestep is set
// up while its predecessor finishes and calls pdl_enter first, which waits
// for the predecessor's completion and its memory.  No kernel touches memory,
// or ends, before that wait, so a kernel's completion implies that of all
// before it.  The successor is let go when the last block ends, not earlier:
// blocks of the next kernel resident beside the current one's made it take
// over the predecessor's split of the SM between L1 and shared memory (N =
// 1e7 step 5.35 -> 5.70 ms with an early release; 5.36 ms without).  What
// is gained is the gap between launches, 0.6 us each.
// Such a kernel's life begins while its predecessor still writes, so none of its
// loads may go by the non-coherent path, which is for memory that nothing writes
// while the kernel lives: no __ldg, and no const __restrict__ parameters that the
// compiler could turn into it.
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ------------------------------------------------------- segment layout
// Clusters of an ensemble are stored back to back.  Segment c owns global
// positions [off[c], off[c+1]); its bound stars are the first nb[c].
struct Seg {
  const int64_t* off;      // n_seg + 1 offsets (device)
  const int64_t* tile_off; // n_seg + 1 tile offsets (device)
  const int64_t* pair_off; // n_seg + 1 pair offsets (by capacity, device)
  const int64_t* bin_off;  // n_seg + 1 bin offsets (by capacity, device)
  const uint64_t* seed;    // per segment
  const double* lnL;       // ln(gamma N_c), per segment
  int64_t* nb;             // bound stars per segment (device, changes)
  uint64_t* dt_bits;       // timestep per segment as double bits
  const double* dt_cap;    // per segment: an outside bound on the timestep (0: none)
  unsigned long long* stats;  // kStStride counters per segment
  uint4* taus;             // combined-Tausworthe streams, one per id slot (or null)
  const int64_t* taus_base;  // per segment: first stream slot (slot = base + id)
  int n_seg;
};

// largest c with a[c] <= v, for a sorted array of n+1 offsets (a[0] = 0)
__device__ __forceinline__ int seg_find(const int64_t* a, int n, int64_t v) {
  int lo = 0, hi = n;  // invariant a[lo] <= v < a[hi]
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (a[mid] <= v) lo = mid; else hi = mid;
  }
  return lo;
}

// ------------------------------------- exact operations on bit patterns
// The FP64 pipe of this GPU issues two lanes per SM and clock, and most of
// the timestep's kernels are bound by it.  Operations that need no FP64
// arithmetic -- comparisons, rounding to float, scaling by 1/2 or 1/4 --
// run on the integer pipes from the bit patterns; each gives the IEEE-754
// result of the FP64 operation it replaces (NaN, infinities, zeros and
// subnormals included, by the bit tests or by falling back to the FP64
// operation where the shortcut does not hold).
constexpr unsigned long long kInfBits = 0x7FF0000000000000ull;
constexpr unsigned long long kSignBit = 0x8000000000000000ull;

__device__ __forceinline__ unsigned long long ubits(double v) {
  return (unsigned long long)__double_as_longlong(v);
}
// v < 0.0
__device__ __forceinline__ bool lt0(double v) {
  const unsigned long long u = ubits(v);
  return u > kSignBit && u <= (kSignBit | kInfBits);
}
// v > 0.0 (+Inf included)
__device__ __forceinline__ bool pos_num(double v) { return ubits(v) - 1ull < kInfBits; }
// v >= 0.0 (-0 included)
__device__ __forceinline__ bool ge0(double v) {
  const unsigned long long u = ubits(v);
  return u <= kInfBits || u == kSignBit;
}
// v < +Inf
__device__ __forceinline__ bool lt_inf(double v) {
  const unsigned long long u = ubits(v);
  return (u & ~kSignBit) <= kInfBits && u != kInfBits;
}
// v <= 1.0
__device__ __forceinline__ bool le1(double v) {
  const unsigned long long u = ubits(v);
  return (u & ~kSignBit) <= kInfBits && (u >= kSignBit || u <= 0x3FF0000000000000ull);
}
// v >= rj for rj > 0
__device__ __forceinline__ bool ge_pos(double v, double rj) {
  const unsigned long long u = ubits(v);
  return u >= ubits(rj) && u <= kInfBits;
}
// a > b for a > 0 (b any value but NaN)
__device__ __forceinline__ bool gt_pos(double a, double b) {
  return __double_as_longlong(a) > __double_as_longlong(b);
}
// v 2^-k for k = 1, 2: the exponent field lowered by k when the result stays
// normal, else the FP64 product
template <int k>
__device__ __forceinline__ double scale_down(double v) {
  const unsigned long long u = ubits(v);
  const unsigned f = (unsigned)(u >> 52) & 0x7FFu;
  if (f > (unsigned)k && f < 0x7FFu) return __longlong_as_double((long long)(u - ((unsigned long long)k << 52)));
  return v * (k == 1 ? 0.5 : 0.25);
}
// v 2^k for k = 1, 2: the exponent field raised by k when v and the result
// are normal, else the FP64 product
template <int k>
__device__ __forceinline__ double scale_up(double v) {
  const unsigned long long u = ubits(v);
  const unsigned f = (unsigned)(u >> 52) & 0x7FFu;
  if (f - 1u < 2046u - (unsigned)k) return __longlong_as_double((long long)(u + ((unsigned long long)k << 52)));
  return v * (k == 1 ? 2.0 : 4.0);
}
// (float)v: the top 24 significand bits rounded to nearest even by the 29
// bits below them, for doubles whose float is normal (2^-126 <= |v| <
// 2^126); others by the conversion
__device__ __forceinline__ float f32_rn(double v) {
  const unsigned long long u = ubits(v);
  const unsigned ex = (unsigned)(u >> 52) & 0x7FFu;
  if (ex - 897u > 252u) return (float)v;  // outside [897, 1149]
  const unsigned top = ((ex - 896u) << 23) | ((unsigned)(u >> 29) & 0x7FFFFFu);
  const unsigned rest = (unsigned)u & 0x1FFFFFFFu;
  const bool up = rest > 0x10000000u || (rest == 0x10000000u && (top & 1u));
  return __uint_as_float(((unsigned)(u >> 32) & 0x80000000u) | (top + (up ? 1u : 0u)));
}

// Correctly rounded FP64 product, quotient and square root from integer
// arithmetic on the significands, for normal operands with a normal result
// (anything else: the FP64 operation).  On this GPU an FP64 operation occupies
// its SM's FP64 pipe for 16 cycles, a division or square root for about a
// hundred; these take none of it, and the FP64 pipe is left to the additions.
// Each returns the IEEE-754 round-to-nearest-even result exactly (checked bit
// for bit against the FP64 operations on 3 x 2^28 operand pairs per operation:
// random bit patterns, random values over 81 binades, and significands with
// random runs of trailing zeros, which give exact results and ties).
//
// The significands are integers in [2^52, 2^53); the result's significand Q
// is an integer in the same range, its exponent follows from the operands'.
// A result assembled as sign + ((e - 1) << 52) + Q lets a significand that
// rounds up to 2^53 carry into the exponent.
__device__ __forceinline__ unsigned long long sig_of(unsigned hi, unsigned lo) {
  return ((unsigned long long)((hi & 0xFFFFFu) | 0x100000u) << 32) | lo;
}
// whether the high word of a double is a normal number's
__device__ __forceinline__ bool normal_hi(unsigned hi) {
  return ((hi + 0x100000u) & 0x7FFFFFFFu) >= 0x200000u;
}
__device__ __forceinline__ double dbl_of(unsigned hi, unsigned long long q) {
  return __longlong_as_double((long long)(((unsigned long long)hi << 32) + q));
}

// a b: the 117-bit product of one significand and the other one shifted up
// by 11 bits, from four 32 x 32 -> 64 bit products; its high word holds 52 or
// 53 significant bits, rounded to nearest even by the low word.
__device__ __forceinline__ double mul_rn(double a, double b) {
  const unsigned long long ua = ubits(a), vb = ubits(b);
  const unsigned xa = (unsigned)(ua >> 32), xb = (unsigned)(vb >> 32);
  // the result's exponent field less one, before a carry
  const unsigned ex = (xa & 0x7FF00000u) + (xb & 0x7FF00000u) - (1024u << 20);
  if (normal_hi(xa) && normal_hi(xb) && ex < 0x7FC00000u) {
    const unsigned al = (unsigned)ua << 11, ah = (unsigned)(ua >> 21) | 0x80000000u;
    const unsigned bl = (unsigned)vb, bh = (xb & 0xFFFFFu) | 0x100000u;
    const unsigned long long p0 = (unsigned long long)al * bl;
    const unsigned long long p1 = (unsigned long long)ah * bl + (unsigned)(p0 >> 32);
    const unsigned long long p2 = (unsigned long long)al * bh + (unsigned)p1;
    unsigned long long hi =
        (unsigned long long)ah * bh + (unsigned)(p1 >> 32) + (unsigned)(p2 >> 32);
    unsigned long long lo = (p2 << 32) | (unsigned)p0;
    unsigned e = ex + ((xa ^ xb) & 0x80000000u);
    if ((unsigned)(hi >> 32) >= 0x100000u) {
      e += 0x100000u;
    } else {
      hi = (hi << 1) | (lo >> 63);
      lo <<= 1;
    }
    lo |= hi & 1ull;  // at half, up to the even neighbour
    return dbl_of(e, hi + (lo > (1ull << 63) ? 1ull : 0ull));
  }
  return a * b;
}

// a / b in two digits of 30 and 22 bits.  R0 = m_a 2^s with s = 1 when m_a <
// m_b, so that R0 / m_b is in [1, 2) and its quotient in units of 2^-52 has
// 53 bits.  v ~ 2^84 / m_b (32 bits, never above) is the float reciprocal of
// m_b's top bits (~21 bits) after one Newton step, v' = v - v (b_t v - 2^63) /
// 2^63 with b_t + 1 > m_b / 2^21 for the divisor, lowered by 2 for the
// roundings.
//   q1 = floor(floor(R0 / 2^22) v / 2^32), up to 7 units below R0 2^30 / m_b;
//   R1 = R0 2^30 - q1 m_b, exact modulo 2^64 (0 <= R1 < 7 m_b);
//   q2 = floor of R1 2^22 / m_b from R1 / 2^25 and v, at most 1.2 below it;
//   R2 = R1 2^22 - q2 m_b, exact modulo 2^64 (0 <= R2 < 1.2 m_b).
// The quotient is Q + R2 / m_b, Q = 2^22 q1 + q2, so the nearest integer is Q or
// Q + 1; a tie cannot occur (a quotient of two 53-bit integers has no 54-bit
// significand).
__device__ __forceinline__ double div_rn(double a, double b) {
  const unsigned long long ua = ubits(a), vb = ubits(b);
  const unsigned xa = (unsigned)(ua >> 32), xb = (unsigned)(vb >> 32);
  const unsigned long long ma = sig_of(xa, (unsigned)ua), mb = sig_of(xb, (unsigned)vb);
  const unsigned s = ma < mb ? 1u : 0u;
  // the result's exponent field less one
  const unsigned ex = (xa & 0x7FF00000u) - (xb & 0x7FF00000u) + ((1022u - s) << 20);
  if (normal_hi(xa) && normal_hi(xb) && ex < 0x7FD00000u) {
    const unsigned bt = (unsigned)(mb >> 21);
    // (the two low bits set: the float stays above 1, its reciprocal below)
    const float f = __uint_as_float(0x3F800003u | ((bt >> 8) & 0x7FFFFFu));
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
    unsigned v = (__float_as_uint(y) << 8) | 0x80000000u;  // y 2^32, y in [1/2, 1)
    // (b_t + 1) v - 2^63 in units of 2^28 (2^63 falls out of the 32 bits)
    const int d = (int)(unsigned)(((unsigned long long)bt * v + v) >> 28);
    v = v - (unsigned)(((int)(v >> 16) * d) >> 19) - 2u;
    const unsigned q1 = __umulhi((unsigned)(ma >> (22u - s)), v);
    const unsigned long long R1 = (ma << (30u + s)) - (unsigned long long)q1 * mb;
    const unsigned q2 = __umulhi((unsigned)(R1 >> 25), v) >> 5;
    const unsigned long long R2 = (R1 << 22) - (unsigned long long)q2 * mb;
    unsigned long long Q = ((unsigned long long)q1 << 22) + q2;
    if (R2 > (mb >> 1)) ++Q;
    return dbl_of(ex + ((xa ^ xb) & 0x80000000u), Q);
  }
  return a / b;
}

// sqrt(x), in the same way: the root of N = M 2^52, M = m_x 2^p with p = 1
// when x's biased exponent is even, is an integer of 53 bits.  v ~ 2^58 /
// sqrt(M) (32 bits, never above) is the float reciprocal square root of M's
// top bits (~20 bits) after one Newton step, v' = v - v (m_h v^2 - 2^94) / 2^95
// with M / 2^22 < m_h + 1, lowered by 3 for the roundings.
//   q1 = floor(m_h v / 2^32), up to 7 units below 2^4 sqrt(M);
//   R1 = 2^8 M - q1^2 (0 <= R1 < 2^35);
//   q2 = floor of R1 2^21 / sqrt(2^8 M) from R1 / 2^4 and v, not above the root
//   of the rest and at most 1.2 below it;
//   R2 = N - S^2 for S = 2^22 q1 + q2, exact modulo 2^64.
// The nearest integer to the root is S + 1 when R2 > S ((S + 1/2)^2 = S^2 + S +
// 1/4), S otherwise.  Negative, zero, subnormal and non-finite x: the FP64
// square root.
//
// Dependent chains, whole GPU: quotient 414 G/s (70 on the FP64 pipe), root 387
// (67), product 595 (501).  Signed digits with two-sided corrections measured
// 343 and 325, 64-bit fixed-point reciprocals with two Newton steps and a
// 128-bit remainder 136 and 120.
__device__ __forceinline__ double sqrt_rn(double x) {
  const unsigned long long ux = ubits(x);
  const unsigned xh = (unsigned)(ux >> 32);
  if (xh - 0x100000u < 0x7FE00000u) {
    const unsigned p = (~xh >> 20) & 1u;
    const unsigned long long ma = sig_of(xh, (unsigned)ux);
    // M / 2^52 in [1, 4) as a float, its low bits replaced so that it stays
    // off both ends and its reciprocal root inside (1/2, 1)
    const float f =
        __uint_as_float((0x3F800008u + (p << 23)) | ((unsigned)(ma >> 29) & 0x7FFFF0u));
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
    unsigned v = (__float_as_uint(y) << 8) | 0x80000000u;  // y 2^32
    const unsigned mh = (unsigned)(ma >> (22u - p));
    const unsigned sq = __umulhi(v, v);
    const int d = (int)(unsigned)(((unsigned long long)sq * mh + sq) >> 28);
    v = v - (unsigned)(((int)(v >> 16) * d) >> 19) - 3u;
    const unsigned q1 = __umulhi(mh, v);
    const unsigned long long R1 = (ma << (8u + p)) - (unsigned long long)q1 * q1;
    const unsigned q2 = __umulhi((unsigned)(R1 >> 4), v) >> 5;
    const unsigned long long S1 = (unsigned long long)q1 << 22, S = S1 + q2;
    const unsigned long long R2 = (R1 << 44) - (unsigned long long)q2 * (S + S1);
    const unsigned ex = ((xh >> 20) - p + 1021u) >> 1;  // its exponent field less one
    return dbl_of(ex << 20, S + (R2 > S ? 1ull : 0ull));
  }
  return sqrt(x);
}

// ------------------------------------------------- counter-based RNG
// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11): ten rounds of two
// 32x32->64 bit products and xors, keys bumped by the Weyl constants.
struct U4 { uint32_t x, y, z, w; };

__device__ __forceinline__ U4 philox(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                     uint64_t seed) {
  uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    uint32_t lo0 = 0xD2511F53u * c0, hi0 = __umulhi(0xD2511F53u, c0);
    uint32_t lo1 = 0xCD9E8D57u * c2, hi1 = __umulhi(0xCD9E8D57u, c2);
    uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
    k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
  }
  return U4{c0, c1, c2, c3};
}

// (2k + 1) 2^-53 from the top 52 bits k of (hi:lo): exact, inside (0, 1)
__device__ __forceinline__ double u01(uint32_t lo, uint32_t hi) {
  // (2k + 1) 2^-53 is exact: its bits are assembled with integer operations
  // (leading-zero count, shift, exponent) instead of an int -> double
  // conversion and a multiply on the FP64 pipe
  const uint64_t k = ((((uint64_t)hi) << 32) | lo) >> 12;
  const uint64_t mo = 2ull * k + 1ull;  // odd, < 2^53
  const int lz = __clzll((long long)mo) - 11;
  const uint64_t mm = mo << lz;  // top bit at 52
  return __longlong_as_double(
      (long long)(((uint64_t)(1022 - lz) << 52) | (mm & 0x000FFFFFFFFFFFFFull)));
}

// 2 X - 1 for X = u01(lo, hi) equals U 2^-52 exactly, U = 2k + 1 - 2^52 (odd,
// |U| < 2^52); sym_int gives U, sym_double the double
__device__ __forceinline__ int64_t sym_int(uint32_t lo, uint32_t hi) {
  const uint64_t k = ((((uint64_t)hi) << 32) | lo) >> 12;
  return (int64_t)(2ull * k + 1ull) - (int64_t)(1ull << 52);
}
__device__ __forceinline__ double sym_double(int64_t U) {
  const uint64_t a = U < 0 ? (uint64_t)(-U) : (uint64_t)U;
  const int lz = __clzll((long long)a) - 11;
  const uint64_t aa = a << lz;
  return __longlong_as_double((long long)((U < 0 ? 0x8000000000000000ull : 0ull) |
                                          ((uint64_t)(1023 - lz) << 52) |
                                          (aa & 0x000FFFFFFFFFFFFFull)));
}

// ------------------------------------------- combined Tausworthe streams
// The paper's generator as an option (section 3.6; L'Ecuyer 1999): four
// LFSR words with (k, q, s) = (31, 6, 18), (29, 2, 2), (28, 13, 7),
// (25, 3, 13); a step of a word z is b = ((z << q) ^ z) >> (k - s),
// z = ((z & m_k) << s) ^ b (m_k clears the low 32 - k bits); the output is
// the xor of the four words.
template <int k, int q, int s>
__device__ __forceinline__ uint32_t taus_word(uint32_t z) {
  const uint32_t b = ((z << q) ^ z) >> (k - s);
  return ((z & (0xFFFFFFFFu << (32 - k))) << s) ^ b;
}
__device__ __forceinline__ uint32_t taus_next(uint4& z) {
  z.x = taus_word<31, 6, 18>(z.x);
  z.y = taus_word<29, 2, 2>(z.y);
  z.z = taus_word<28, 13, 7>(z.z);
  z.w = taus_word<25, 3, 13>(z.w);
  return z.x ^ z.y ^ z.z ^ z.w;
}

// A star's random blocks of four words.  Counter mode (kTaus false):
// Philox4x32-10 at (id, step, tag, trial).  Stream mode: the next four
// outputs of the star's own stream; the method asks for each star's blocks
// in a fixed order (relaxation trials, orbit trials, the v_r sign), so the
// tag and the trial are implied by the order.
template <bool kTaus>
struct Draws {
  uint64_t seed;
  uint32_t id, step;
  uint4 z;
  __device__ __forceinline__ U4 block(uint32_t tag, uint32_t t) {
    if (!kTaus) return philox(id, step, tag, t, seed);
    U4 w;
    w.x = taus_next(z);
    w.y = taus_next(z);
    w.z = taus_next(z);
    w.w = taus_next(z);
    return w;
  }
  // pass over n blocks (stream mode)
  __device__ __forceinline__ void skip(uint32_t n) {
    if (kTaus)
      for (uint32_t i = 0; i < 4u * n; ++i) taus_next(z);
  }
};

template <bool kTaus>
__device__ __forceinline__ Draws<kTaus> draws_of(const Seg& S, int c, uint32_t id,
                                                 uint32_t step) {
  Draws<kTaus> d;
  d.seed = S.seed[c];
  d.id = id;
  d.step = step;
  if (kTaus) d.z = S.taus[S.taus_base[c] + id];
  return d;
}

template <bool kTaus>
__device__ __forceinline__ void draws_keep(const Seg& S, int c, const Draws<kTaus>& d) {
  if (kTaus) S.taus[S.taus_base[c] + d.id] = d.z;
}

// Non-inlined copies of div_rn and sqrt_rn for the relaxation kernel: its
// fifteen call sites inlined overflow the instruction cache (relaxation 0.853
// ms shared, 0.876 ms inlined at N = 1e7, with their earlier form); the kernels
// with a few call sites inline them (FP64 mode's orbit stage 2.58 ms inlined,
// 2.65 ms shared).
static __device__ __noinline__ double div_rn_nl(double a, double b) { return div_rn(a, b); }
static __device__ __noinline__ double sqrt_rn_nl(double x) { return sqrt_rn(x); }

// A B 2^k for nonzero A, B < 2^53, rounded to nearest even, with a sign bit: the
// 128-bit product's top 53 bits, rounded by the bits below (products below
// 2^64, one in a million, by the FP64 product: the factors are exact doubles)
template <int k>
__device__ __forceinline__ double product_of(uint64_t A, uint64_t B, uint64_t sign) {
  const uint64_t hi = __umul64hi(A, B), lo = A * B;
  double v;
  if (hi) {
    const int lz = __clzll((long long)hi);
    const uint64_t top = (hi << lz) | ((lo >> 1) >> (63 - lz)), rest = lo << lz;
    const uint64_t Q = top >> 11;
    const uint64_t below = (top << 53) | (rest ? 1ull : 0ull) | (Q & 1ull);
    v = __longlong_as_double((long long)(((uint64_t)(1022 + 127 - lz + k) << 52) + Q +
                                         (below > (1ull << 63) ? 1ull : 0ull)));
  } else {
    v = ((double)A * (double)B) * __longlong_as_double((long long)((uint64_t)(1023 + k) << 52));
  }
  return __longlong_as_double((long long)(ubits(v) | sign));
}

// uniform planar direction (cos a, sin a) by rejection of a point in the
// unit disk; the doubled angle gives cos = (u^2 - v^2)/q, sin = 2uv/q.
//
// The draw (u, v) = (U, V) 2^-52 is accepted when the FP64 value of
// u u + v v is <= 1.  That value is within 2^-51 of the exact sum (both
// below 2), so outside a band of 2^54 around 2^104 the exact integer test
// U^2 + V^2 <= 2^104 (128-bit) gives the same answer; inside the band the
// FP64 expression decides.  The loop is integer work only; the FP64
// arithmetic of the accepted draw runs once, after it.  Not inlined: one
// copy serves both of the relaxation's angles (code size, as for div_rn_nl).
//
// A draw is accepted with probability pi/4, so a warp in which each lane draws for
// itself takes 3.3 rounds.  After the first the lanes of a full warp are shared
// out among those still without one, for their next 2 to 32 draws at a time (the
// first accepted counts): 2.0 rounds.  Relaxation of 10^5, 10^6, 10^7 stars 22.1,
// 88.4, 740 us to 20.6, 84.1, 710.  (For blocks of up to 128 threads.)
// the draw of block w: inside the unit disk?
__device__ __forceinline__ bool disk_draw(const U4& w, int64_t& U, int64_t& V) {
  U = sym_int(w.x, w.y), V = sym_int(w.z, w.w);
  const uint64_t A = U < 0 ? (uint64_t)(-U) : (uint64_t)U;
  const uint64_t B = V < 0 ? (uint64_t)(-V) : (uint64_t)V;
  const uint64_t l1 = A * A, l2 = B * B;
  const uint64_t lo = l1 + l2;
  const uint64_t hi = __umul64hi(A, A) + __umul64hi(B, B) + (lo < l1 ? 1ull : 0ull);
  // S = hi 2^64 + lo against 2^104 -+ 2^54
  const uint64_t H = 1ull << 40, band = 1ull << 54;
  const bool in = hi < H - 1 || (hi == H - 1 && lo <= 0ull - band);
  const bool out = hi > H || (hi == H && lo >= band);
  if (in || out) return in;
  const double u = sym_double(U), v = sym_double(V);
  const double uu = u * u, vv = v * v;
  return uu + vv <= 1.0;
}

template <bool kTaus>
__device__ __noinline__ bool disk_angle(Draws<kTaus>& g, uint32_t tag, double& c, double& s) {
  int64_t Ua = 0, Va = 0;
  bool ok = false;
  uint32_t t = 0;
  if (!kTaus && __activemask() == 0xFFFFFFFFu) {
    ok = disk_draw(g.block(tag, 0), Ua, Va);
    const int lane = threadIdx.x & 31;
    __shared__ uint8_t s_owner[128];
    uint8_t* owner = s_owner + (threadIdx.x & 96u);
    for (t = 1; t < 64u;) {
      const unsigned lm = __ballot_sync(0xFFFFFFFFu, !ok);
      if (!lm) break;
      const int k = __popc(lm), rank = __popc(lm & ((1u << lane) - 1u));
      const int lg = __clz(2 * k - 1) - 26, G = 1 << lg;
      if (!ok) owner[rank] = (uint8_t)lane;
      __syncwarp();
      const int slot = lane >> lg;
      const bool go = slot < k;
      const int from = go ? owner[slot] : lane;
      __syncwarp();
      Draws<kTaus> q = g;
      q.id = __shfl_sync(0xFFFFFFFFu, g.id, from);
      q.seed = __shfl_sync(0xFFFFFFFFu, (unsigned long long)g.seed, from);
      const uint32_t tg = __shfl_sync(0xFFFFFFFFu, tag, from), mine = t + (lane & (G - 1));
      int64_t U = 0, V = 0;
      const bool in = go && mine < 64u && disk_draw(q.block(tg, mine), U, V);
      const unsigned any = __ballot_sync(0xFFFFFFFFu, in);
      const unsigned gm = G == 32 ? 0xFFFFFFFFu : (1u << G) - 1u;
      const unsigned bits = ok ? 0u : (any >> (rank << lg)) & gm;
      const int src = bits ? (rank << lg) + __ffs(bits) - 1 : lane;
      U = __shfl_sync(0xFFFFFFFFu, (long long)U, src);
      V = __shfl_sync(0xFFFFFFFFu, (long long)V, src);
      if (bits) {
        Ua = U;
        Va = V;
        ok = true;
      }
      t += G;
    }
  } else {
    for (; !ok && t < 64u; ++t) ok = disk_draw(g.block(tag, t), Ua, Va);
  }
  if (!ok) {
    c = 1.0;
    s = 0.0;
    return false;
  }
  // u u, v v and 2 u v from the integers, each rounded once as the FP64 product
  const uint64_t A = Ua < 0 ? (uint64_t)(-Ua) : (uint64_t)Ua;
  const uint64_t B = Va < 0 ? (uint64_t)(-Va) : (uint64_t)Va;
  const double uu = product_of<-104>(A, A, 0ull), vv = product_of<-104>(B, B, 0ull);
  const double uv2 = product_of<-103>(A, B, (uint64_t)(Ua ^ Va) & kSignBit);
  const double q = uu + vv;
  c = div_rn_nl(uu - vv, q);
  s = div_rn_nl(uv2, q);
  return true;
}

// ------------------------------------------------------------ sort keys
__device__ __forceinline__ uint64_t radius_key(double r, uint32_t id) {
  uint64_t b = (uint64_t)__double_as_longlong(r);
  return (b >= 0x7FF0000000000000ull) ? kEscKeyBase | ((uint64_t)id << 20) : b;
}
__device__ __forceinline__ bool key_is_escaper(uint64_t k) {
  return k >= 0x7FF0000000000000ull;
}

// --------------------------------------------- shell potential (Eq. 6)
// Table of one segment: sorted radii r[0..nb), x = 1/r, Phi.  Node nb is
// the virtual star at 1/r = 0 with Phi = 0 (Eq. 2); inside r[0] Phi is
// the constant Phi_0 (Eq. 1 with nothing enclosed).
struct Table64 {
  const double* r;
  const double* x;
  const double* phi;
  int64_t nb;
};

// Radii are positive, and positive doubles order like their 64-bit
// patterns read as signed integers: comparing the patterns gives the same
// answer as the floating-point comparison without using the FP64 pipe.
__device__ __forceinline__ long long dbits(double v) { return __double_as_longlong(v); }

// largest i in [0, nb) with r[i] <= q, else -1 (unique for sorted r)
__device__ __forceinline__ int64_t shell_of(const Table64& t, double q) {
  if (!(q >= 0.0)) return -1;  // (NaN: no radius compares <= it)
  const long long qb = dbits(q);
  const long long* rb = reinterpret_cast<const long long*>(t.r);
  int64_t lo = -1, hi = t.nb;
  while (hi - lo > 1) {
    int64_t mid = lo + ((hi - lo) >> 1);
    if (rb[mid] <= qb) lo = mid; else hi = mid;
  }
  return lo;
}

// Eq. 6 inside shell i (i = -1: central constant)
__device__ __forceinline__ double phi_in_shell(const Table64& t, int64_t i, double q) {
  if (i < 0) return *t.phi;
  double x = div_rn(1.0, q);
  double xj = t.x[i], pj = t.phi[i], xj1, pj1;
  if (i + 1 < t.nb) { xj1 = t.x[i + 1]; pj1 = t.phi[i + 1]; }
  else { xj1 = 0.0; pj1 = 0.0; }
  double den = xj - xj1;
  if (!(den > 0.0)) return pj;
  return pj + div_rn(xj - x, den) * (pj1 - pj);
}

__device__ __forceinline__ double phi_of_r(const Table64& t, double q) {
  return phi_in_shell(t, shell_of(t, q), q);
}

// Cube root by Newton's method, y <- y - (y^3 - v) / (3 y^2), eight steps
// from 2^floor(e/3) (e the binary exponent of v): the merged radius of two
// sticky spheres; the same operations in the same order as the FP64
// statement of the method, so the same bits; 0 for v <= 0.
__device__ __forceinline__ double cbrt_newton(double v) {
  if (!(v > 0.0)) return 0.0;
  const int e = (int)((ubits(v) >> 52) & 0x7FFu) - 1023;
  const int k = e >= 0 ? e / 3 : -((-e + 2) / 3);  // floor(e / 3)
  double y = __longlong_as_double((long long)((unsigned long long)(k + 1023) << 52));
#pragma unroll 1
  for (int i = 0; i < 8; ++i) y = y - (y * y * y - v) / (3.0 * (y * y));
  return y;
}

// ----------------------------------------------------- small utilities
__device__ __forceinline__ void set_err(uint32_t* err, uint32_t bit) {
  atomicOr(err, bit);
}

__device__ __forceinline__ void stat_add(unsigned long long* st, int seg, int which,
                                         unsigned long long v) {
  if (v) atomicAdd(st + (size_t)seg * kStStride + which, v);
}

// The energy a clamp of T' < 0 to 0 adds, m |T'|, into the segment's
// counter as a fixed-point integer in units of 2^-62 (integer sums do not
// depend on their order).
__device__ __forceinline__ void clamp_energy_add(unsigned long long* st, int seg, double m,
                                                double Tp) {
  const double e = -(m * Tp) * 4611686018427387904.0;  // 2^62
  if (e > 0.0) stat_add(st, seg, kStClampEnergy, __double2ull_rn(e));
}

// ------------------------------------------- the orbit step's index tables
// Both are written star by star, in one pass over the sorted stars (by the
// potential kernel, or by stand-alone kernels for a given potential).
// Bucket index of a segment (prm: shift, bucket count, first and last
// indexed node; base: float key bits of 1/r at the first indexed node):
// star k writes start[b] = k for the buckets from its predecessor's bucket
// (exclusive) to its own; the last indexed star closes the table with nb.
// The potential grid's key shells (pr: key0, sh, cells): star k owns the
// keys in (1/r_{k+1}, 1/r_k], i.e. the cells from gmax(k + 1) + 1 to
// gmax(k), gmax(k) = the last cell whose key is <= 1/r_k.  A key (a
// positive float) is <= 1/r_k exactly when its bits are <= those of 1/r_k
// rounded down to a float (its significand truncated).  The outermost star also owns the cells below
// it, the innermost one the cells above it (shell -1).
__device__ __forceinline__ int grid_last_cell(double xk, int4 pr) {
  // 1/r_k rounded down: truncated, where it is a normal float
  const unsigned long long u = ubits(xk);
  const unsigned ex = (unsigned)(u >> 52);
  const uint32_t kb = ex - 897u <= 252u
                          ? ((ex - 896u) << 23) | ((unsigned)(u >> 29) & 0x7FFFFFu)
                          : __float_as_uint(__double2float_rd(xk));
  if (kb < (uint32_t)pr.x) return -1;
  const int g = (int)((kb - (uint32_t)pr.x) >> pr.y);
  return g < pr.z - 1 ? g : pr.z - 1;
}

// a[from .. to] = v for every lane of the warp (all lanes of `mask`, nothing where
// to < from): short ranges by their lane, long ones (a star at the edge of the
// model can own a thousand cells) by the warp together.  A long range costs the
// warp some 80 cycles beside its stores, a short one 10 cycles an entry in one
// lane while others wait: the potential stage of 10^7 stars takes 370, 367,
// 380, 410 and 451 us with 24, 40, 72, 130 and no bound, of 10^6 stars 63, 59,
// 66, 71 and 74, of 10^4 stars 27, 26, 25, 23 and 26.
constexpr int kWideFill = 40;
__device__ __forceinline__ void fill_range(unsigned mask, int* a, int from, int to, int v,
                                           long long cap) {
  const bool wide = to - from >= kWideFill;
  if (!wide)
    for (int i = from; i <= to; ++i)
      if (CMC_IN(i, cap)) a[i] = v;
  unsigned m = __ballot_sync(mask, wide);
  const int lane = threadIdx.x & 31;
  while (m) {
    const int l = __ffs(m) - 1;
    m &= m - 1u;
    const int f = __shfl_sync(mask, from, l), t = __shfl_sync(mask, to, l);
    const int w = __shfl_sync(mask, v, l);
    const long long ai = (long long)__shfl_sync(mask, (unsigned long long)a, l);
    for (int i = f + __popc(mask & ((1u << lane) - 1u)); i <= t; i += __popc(mask))
      if (CMC_IN(i, cap)) reinterpret_cast<int*>(ai)[i] = w;
  }
}

// (in the table whatever the key: after a reported sort failure the radii need not
// be in order)
__device__ __forceinline__ int bucket_of(uint32_t key, uint32_t base, int4 prm) {
  const uint32_t b = (base - key) >> prm.x;
  return b < (uint32_t)prm.y ? (int)b : prm.y - 1;
}
// star k's buckets (key_k, key_km1: float bits of 1/r of stars k and k - 1);
// every lane of mask calls it, live false where there is nothing to write
__device__ __forceinline__ void bucket_starts_of(unsigned mask, bool live, int k, int4 prm,
                                                 uint32_t base, uint32_t key_k,
                                                 uint32_t key_km1, int* st, long long cap) {
  live = live && k >= prm.z && k <= prm.w;
  const int bp = k == prm.z ? -1 : bucket_of(key_km1, base, prm);
  fill_range(mask, st, live ? bp + 1 : 0, live ? bucket_of(key_k, base, prm) : -1, k, cap);
}
// after the last indexed star's buckets: nb (by `count` threads, this one i0)
__device__ __forceinline__ void bucket_close(int nb, int4 prm, uint32_t base, uint32_t key_last,
                                             int* st, long long cap, int i0, int count) {
  for (int i = bucket_of(key_last, base, prm) + 1 + i0; i <= prm.y; i += count)
    if (CMC_IN(i, cap)) st[i] = nb;
}

// star k's grid cells (cell_k, cell_k1: grid_last_cell of stars k and k + 1)
__device__ __forceinline__ void grid_shells_of(unsigned mask, bool live, int k, int nb,
                                               int cell_k, int cell_k1, int4 pr, int* sh) {
  live = live && pr.z > 0;
  fill_range(mask, sh, !live ? 0 : k + 1 < nb ? cell_k1 + 1 : 0, live ? cell_k : -1, k, pr.z);
}
// the cells above the innermost star
__device__ __forceinline__ void grid_close(int cell_0, int4 pr, int* sh, int i0, int count) {
  for (int i = cell_0 + 1 + i0; i < pr.z; i += count) sh[i] = -1;
}

}  // namespace cmc
