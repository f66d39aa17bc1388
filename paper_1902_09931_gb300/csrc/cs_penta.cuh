// The Cahn-Hilliard line solver: (I + a D4) x = b along periodic or reflected lines, the fourth
// difference's pentadiagonal system, in 64-bit fixed point on the integer pipe.
//
// GB300 issues FP64 at 1/64 of the FP32 rate, so an FP64 recursion of the minimal nine operations a
// point is FP64-bound (0.64 ms for both directions at 4096^2; 0.40 ms in fixed point).  A 64 x 64-bit
// fixed-point product is three 32 x 32 -> 64 multiply-adds, so the same recursion on the integer pipes
// costs about a fifth of that, and it rounds at a fixed 2^-53 of the line chunk's largest right-hand
// side or better, where FP64 rounds every partial sum (which grows to ~sqrt(a) times the
// right-hand side) at 2^-53 of itself.
//
// Factorisation.  The operator's symbol is c (1 + p z + q z^2)(1 + p / z + q / z^2) with, for
// g = sqrt((1 + sqrt(1 + 16 a)) / 2) >= 1,
//   c = (g (g + 1) / 2)^2,  p = -2 (g - 1) / g,  q = (g - 1) / (g + 1),
// so a line is a forward recursion y_i = b_i - p y_{i-1} - q y_{i-2} and a backward one
// W_i = y_i - p W_{i+1} - q W_{i+2}, x = W / c: constant coefficients, no tables.  Written with the
// differences D_i = y_i - y_{i-1} both are
//   D_i = D_{i-1} + b_i - (eta y_{i-1} + eps D_{i-1}),   y_i = y_{i-1} + D_i,
//   eta = 1 + p + q = 1 / sqrt(c) = 2 / (g (g + 1)),   eps = 1 - q = 2 / (g + 1),
// whose two products have positive coefficients of at most 1 (unsigned arithmetic on biased values).
//
// Partition.  A line of n points is cut into P chunks of m.  Phase 1 runs both recursions on every
// chunk from zero states and keeps four end values: the forward state (y, D) after the chunk and the
// backward state (W, E = W_0 - W_1) before it, scaled by powers of two.  The true states entering every chunk follow from
// these by 2 x 2 matrices (powers of the recursion's own matrix, a scan over the chunks; periodic
// lines close through (I - M^P)^-1, reflected ones through the boundary's mirror conditions).  Phase 2
// adds the four homogeneous responses to those states: x = W / c + sum of 4 table values times 4
// numbers.  Exact up to rounding.
//
// Fixed point.  b is scaled by its chunk's largest exponent so that |y|, |D| < 2^62 whatever the
// data (the host sums the impulse responses' magnitudes); W likewise after a shift of y by s2 bits.
// Chunks whose largest value is outside 2^[-900, 870] take the same recursion in FP64; a value that is not
// finite fills its line with NaN.
// All values live biased by 2^62 (unsigned), coefficients are 64-bit fractions split in 32-bit
// words: a product is hi hi + (lo hi) / 2^32 + (hi lo) / 2^32, two taps share the three accumulators,
// and the accumulators' initial values centre the rounding (the dropped lo lo term's mean included; b
// itself is rounded to nearest), because a bias, or an error with the sign of a slowly varying field, would
// be a drift of the conserved mass.  Zero data stay exactly zero: the
// coefficients are multiples of 4, so the bias's own products are whole numbers.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <vector>

namespace cs {
namespace pn {

constexpr uint64_t kBias = 1ull << 62;     // y, D, W, E
constexpr uint64_t kCoefBias = 1ull << 60;  // table values and the four states of phase 2
constexpr int kMinE = 123, kMaxE = 1893;    // biased exponents of a chunk's largest value for fixed point
constexpr int kNative = -(1 << 30);         // scale mark of a chunk solved in FP64
constexpr int kMaxChunks = 64;

// Everything the kernels take by value.
struct Par {
  uint64_t cn, ce;           // eta, eps times 2^(64 - 2 [wide])
  uint64_t init_a, init_b;   // rounding of the forward pass's accumulators
  uint64_t init_a2;          // of the backward pass (also centres the shift of y)
  uint64_t kc, kc2;          // bias terms of the two passes
  int nb, s2;                // |b| < 2^nb in units of u; W's unit is 2^s2 u
  int levels;                // scan levels whose matrix is not negligible
  int cyclic;                // periodic line whose A^n is negligible: the scan wraps, no closing
  int native;                // a above 1e24: every chunk in FP64
  int wide;                  // small a (g <= 2.25): coefficients scaled by 2^62 instead of 2^64
  uint64_t ic;               // 1 / c = ic 2^(ic_e - 62), ic in [2^61, 2^62)
  int ic_e;
  double eta, eps, inv_c;
  double fs, bs;             // scales of the forward and backward states, the powers of two below 1 / sqrt(c) and 1 / c
  double M[4];               // A^m
  double Ml[6][4];           // A^(m 2^l): the scan's levels
  double R[4];               // backward state before a chunk caused by a unit forward state entering it
  double C[4];               // periodic: (I - A^(mP))^-1
  double V[4];               // reflected: (W, E) after the line from (y, D) at its end
  double Z[4];               // reflected: the forward state entering the line from (W, E) at its start
  uint32_t low[4];           // mean low word of each table
  uint32_t trunc_lo[4], trunc_hi[4];  // 2^31 times the share of points whose low / high word's product is truncated
  int t[4];                  // tables: real value = 2^t (int) / 2^60
};

__host__ __device__ __forceinline__ uint64_t wmul(uint32_t a, uint32_t b) { return static_cast<uint64_t>(a) * b; }
__host__ __device__ __forceinline__ uint32_t hi32(uint64_t v) { return static_cast<uint32_t>(v >> 32); }
__host__ __device__ __forceinline__ uint32_t lo32(uint64_t v) { return static_cast<uint32_t>(v); }

__host__ __device__ __forceinline__ uint64_t dbits(double x) {
#ifdef __CUDA_ARCH__
  return static_cast<uint64_t>(__double_as_longlong(x));
#else
  uint64_t b;
  memcpy(&b, &x, 8);
  return b;
#endif
}
__host__ __device__ __forceinline__ double from_bits(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(static_cast<long long>(b));
#else
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}
// 2^k, k in the normal range
__host__ __device__ __forceinline__ double pow2(int k) { return from_bits(static_cast<uint64_t>(k + 1023) << 52); }

// v >> r, 0 for r >= 64 (PTX clamps the amount)
__host__ __device__ __forceinline__ uint64_t shr(uint64_t v, int r) {
#ifdef __CUDA_ARCH__
  uint64_t o;
  asm("shr.b64 %0, %1, %2;" : "=l"(o) : "l"(v), "r"(r));
  return o;
#else
  return r >= 64 ? 0 : v >> r;
#endif
}

// x 2^(nb - top) as a two's-complement integer (truncated towards zero), for |x| < 2^top and
// E = 64 - nb + 1022 + top; E - (x's biased exponent) is the shift of the left-aligned significand.
// Zeros and subnormals give 0 (E >= 64 for every chunk in fixed point).
__host__ __device__ __forceinline__ uint64_t to_fixed(uint64_t xb, int E) {
  const uint32_t hi = hi32(xb);
  const int e = static_cast<int>((hi >> 20) & 0x7ffu);
  const uint64_t M = (static_cast<uint64_t>((hi & 0xFFFFFu) | 0x100000u) << 32 | lo32(xb)) << 11;
  const uint64_t A = shr(M, E - e);
  const uint64_t s = static_cast<uint64_t>(static_cast<int64_t>(static_cast<int32_t>(hi) >> 31));
  return (A ^ s) - s;
}

// to_fixed to the nearest integer, halves to the even one, on two more bits (E - (x's biased exponent) >= 2).
// Cutting towards zero instead leaves half a unit of x's sign: harmless at a point, but the signs of a
// slowly varying right-hand side stay, and their sum over a line is a drift of the conserved mass (4096^2,
// 1000 steps: twice that of rounding each value).  The bits beyond the two are cut: 1/16 as much.
__host__ __device__ __forceinline__ uint64_t to_fixed_near(uint64_t xb, int E) {
  const uint32_t hi = hi32(xb);
  const int e = static_cast<int>((hi >> 20) & 0x7ffu);
  const uint64_t M = (static_cast<uint64_t>((hi & 0xFFFFFu) | 0x100000u) << 32 | lo32(xb)) << 11;
  const uint64_t A4 = shr(M, E - 2 - e);
  const uint64_t A = (A4 + (((lo32(A4) >> 2) & 1u) + 1u)) >> 2;
  const uint64_t s = static_cast<uint64_t>(static_cast<int64_t>(static_cast<int32_t>(hi) >> 31));
  return (A ^ s) - s;
}

// T 2^e as a double, |T| < 2^62, rounded to nearest (halves away from zero: symmetric in sign).
// The result must be a normal number or zero.
__host__ __device__ __forceinline__ double from_fixed(uint64_t T, int e) {
  const uint64_t s = static_cast<uint64_t>(static_cast<int64_t>(T) >> 63);
  const uint64_t A = (T ^ s) - s;
#ifdef __CUDA_ARCH__
  const int z = __clzll(static_cast<long long>(A));
#else
  const int z = A ? __builtin_clzll(A) : 64;
#endif
  // top bit to bit 62; the rounded significand's leading bit adds one to the exponent field
  const uint64_t m = ((A << ((z - 1) & 63)) + 512u) >> 10;
  const uint64_t b = m + (static_cast<uint64_t>(static_cast<uint32_t>(e + 62 - z + 1 + 1023 - 1)) << 52);
  return from_bits(A ? (b | (s & 0x8000000000000000ull)) : 0ull);
}

// One step of either recursion on biased values: D += b - (eta Y + eps D), Y += D.
template <int WIDE>
__host__ __device__ __forceinline__ void step(uint64_t& Y, uint64_t& D, uint64_t b, uint64_t cn, uint64_t ce,
                                              uint64_t ia, uint64_t ib, uint64_t kc) {
  uint64_t A = wmul(lo32(Y), hi32(cn)) + ia;
  uint64_t B = wmul(hi32(Y), lo32(cn)) + ib;
  uint64_t M = wmul(hi32(Y), hi32(cn));
  A += wmul(lo32(D), hi32(ce));
  B += wmul(hi32(D), lo32(ce));
  M += wmul(hi32(D), hi32(ce));
  M += static_cast<uint64_t>(hi32(A)) + hi32(B);
  D = (D + b + kc) - (WIDE ? M << 2 : M);
  Y = Y + D - kBias;
}

// Phase 1 on one chunk, values at s (an accessor: load8 / store8 move 8 consecutive 64-bit words, get /
// put one; the last m % 8 points are taken one by one).
// Returns the scale mark: the exponent of W's unit, or kNative; ends = (y, D) after the chunk, about divided
// by sqrt(c), and (W, E) before it, about divided by c.  The factors are powers of two, exact, and the
// tables carry the rest: a rounded factor would leave an error in the line's sum that is the same at every
// step for the slowly varying part of the field, a drift of the conserved mass.
template <class Acc>
__host__ __device__ __forceinline__ uint32_t chunk_max_hi(const Acc& s, int m) {
  uint32_t mx = 0;
  for (int k0 = 0; k0 + 8 <= m; k0 += 8) {
    uint64_t v[8];
    s.load8(k0, v);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const uint32_t h = hi32(v[u]) & 0x7fffffffu;
      mx = h > mx ? h : mx;
    }
  }
  for (int k = m & ~7; k < m; ++k) {
    const uint32_t h = hi32(s.get(k)) & 0x7fffffffu;
    mx = h > mx ? h : mx;
  }
  return mx;
}

template <int WIDE, class In, class Acc>
__host__ __device__ __forceinline__ int local_fixed(const Par& q, const In& in, const Acc& s, int m, int te,
                                                    double (&ends)[4]) {
  // te: biased exponent of the chunk's largest value (0: all zero)
  const int E = 64 - q.nb + te;  // |b| < 2^(te - 1022)
  const int eu = te - 1022 - q.nb;  // exponent of y's unit
  uint64_t Y = kBias, D = kBias;
  for (int k0 = 0; k0 + 8 <= m; k0 += 8) {
    uint64_t v[8];
    in.load8(k0, v);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      step<WIDE>(Y, D, to_fixed_near(v[u], E), q.cn, q.ce, q.init_a, q.init_b, q.kc);
      v[u] = Y;
    }
    s.store8(k0, v);
  }
  for (int k = m & ~7; k < m; ++k) {
    step<WIDE>(Y, D, to_fixed_near(in.get(k), E), q.cn, q.ce, q.init_a, q.init_b, q.kc);
    s.put(k, Y);
  }
  ends[0] = static_cast<double>(static_cast<int64_t>(Y - kBias)) * (te ? q.fs * pow2(eu) : 0.0);
  ends[1] = static_cast<double>(static_cast<int64_t>(D - kBias)) * (te ? q.fs * pow2(eu) : 0.0);
  uint64_t W = kBias;
  D = kBias;
  // y in W's unit.  init_a2 makes up for the mean of the bits that the shift drops, except at the chunk's
  // two ends, where y is rounded to nearest even first: at the last point the products from a zero state
  // are exact and make up for nothing, and y of the first point is b itself, whose bits below 2^-53
  // are mostly zero (dropping them lost a quarter of W's unit instead of a half, a bias of 0.016 u a point of
  // x at n = 512).  With wide coefficients D moves in steps of four, so y's low bits are b's at every point:
  // all are rounded (0.23 u a point at n = 64 otherwise).
  auto to_even = [&](uint64_t y) { return q.s2 ? y + ((1ull << (q.s2 - 1)) - 1 + ((y >> q.s2) & 1)) : y; };
  if (!WIDE) {
    s.put(m - 1, to_even(s.get(m - 1)));
    s.put(0, to_even(s.get(0)));
  }
  auto back = [&](uint64_t y, bool first) {
    step<WIDE>(W, D, (WIDE ? to_even(y) : y) >> q.s2, q.cn, q.ce, WIDE || first ? q.init_a : q.init_a2, q.init_b, q.kc2);
    return W;
  };
  for (int k = m - 1; k >= (m & ~7); --k) s.put(k, back(s.get(k), false));
  for (int k0 = (m & ~7) - 8; k0 >= 0; k0 -= 8) {
    uint64_t v[8];
    s.load8(k0, v);
#pragma unroll
    for (int u = 7; u >= 0; --u) v[u] = back(v[u], k0 + u == 0);
    s.store8(k0, v);
  }
  ends[2] = static_cast<double>(static_cast<int64_t>(W - kBias)) * (te ? q.bs * pow2(eu + q.s2) : 0.0);
  ends[3] = static_cast<double>(static_cast<int64_t>(D - kBias)) * (te ? q.bs * pow2(eu + q.s2) : 0.0);
  return te ? eu + q.s2 : -4000;
}

// The same in FP64, for chunks outside fixed point's exponents, on y fs and W bs: W itself is up to c times the
// result and would overflow first.
template <class In, class Acc>
__host__ __device__ __forceinline__ int local_native(const Par& q, const In& in, const Acc& s, int m,
                                                     double (&ends)[4]) {
  double Y = 0.0, D = 0.0;
  for (int k0 = 0; k0 + 8 <= m; k0 += 8) {
    uint64_t v[8];
    in.load8(k0, v);
#pragma unroll 1
    for (int u = 0; u < 8; ++u) {
      D = D + (from_bits(v[u]) * q.fs - fma(q.eta, Y, q.eps * D));
      Y = Y + D;
      v[u] = dbits(Y);
    }
    s.store8(k0, v);
  }
  for (int k = m & ~7; k < m; ++k) {
    D = D + (from_bits(in.get(k)) * q.fs - fma(q.eta, Y, q.eps * D));
    Y = Y + D;
    s.put(k, dbits(Y));
  }
  ends[0] = Y;
  ends[1] = D;
  const double to_w = q.bs / q.fs;  // a power of two
  double W = 0.0;
  D = 0.0;
  for (int k = m - 1; k >= (m & ~7); --k) {
    D = D + (from_bits(s.get(k)) * to_w - fma(q.eta, W, q.eps * D));
    W = W + D;
    s.put(k, dbits(W));
  }
  for (int k0 = (m & ~7) - 8; k0 >= 0; k0 -= 8) {
    uint64_t v[8];
    s.load8(k0, v);
#pragma unroll 1
    for (int u = 7; u >= 0; --u) {
      D = D + (from_bits(v[u]) * to_w - fma(q.eta, W, q.eps * D));
      W = W + D;
      v[u] = dbits(W);
    }
    s.store8(k0, v);
  }
  ends[2] = W;
  ends[3] = D;
  return kNative;
}

// in: the right-hand side's chunk; s: where W goes (may be the same words).
template <class In, class Acc>
__host__ __device__ __forceinline__ int local_solve(const Par& q, const In& in, const Acc& s, int m,
                                                    double (&ends)[4]) {
  const uint32_t mx = chunk_max_hi(in, m);
  const int te = static_cast<int>(mx >> 20);
  if (te == 0x7ff) {  // a non-finite value: the whole line is filled from its end values (correct_chunk)
    ends[0] = ends[1] = ends[2] = ends[3] = from_bits(0x7ff8000000000000ull);
    return kNative;
  }
  if (q.native || (te != 0 && (te < kMinE || te > kMaxE))) return local_native(q, in, s, m, ends);
  return q.wide ? local_fixed<1>(q, in, s, m, te, ends) : local_fixed<0>(q, in, s, m, te, ends);
}

// ---- the states entering the chunks ----------------------------------------------------------------
// o = M v + w (2 x 2, row-major), rounded in a fixed order
__host__ __device__ __forceinline__ void mv_add(const double* M, double v0, double v1, double w0, double w1,
                                                double& o0, double& o1) {
  const double a = fma(M[0], v0, fma(M[1], v1, w0));
  const double b = fma(M[2], v0, fma(M[3], v1, w1));
  o0 = a;
  o1 = b;
}

// ---- phase 2 ---------------------------------------------------------------------------------------
// tab[2 k], tab[2 k + 1]: the four biased table values of point k; base[k]: minus the product of the
// four with the states' own bias.
struct TabRow { uint64_t v[4]; };

// a b / 2^32 + c on 32-bit words
__host__ __device__ __forceinline__ uint32_t mad_hi(uint32_t a, uint32_t b, uint32_t c) {
#ifdef __CUDA_ARCH__
  uint32_t r;
  asm("mad.hi.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
#else
  return hi32(wmul(a, b)) + c;
#endif
}

// The per-chunk constants of phase 2: W's multiplier and the four states, all in output units 2^eo.
// The cross products keep only their high words (one 32-bit multiply-add each; the ten of them fit in
// two 32-bit sums); init makes up for their truncation on average.
struct Corr {
  uint64_t cw, u[4], k0, init;
  int eo;
};

__host__ __device__ __forceinline__ int bexp(double x) { return static_cast<int>((hi32(dbits(x)) >> 20) & 0x7ffu); }

// False when phase 2 has to run in FP64 (states or chunk outside fixed point's exponents).
__host__ __device__ __forceinline__ bool corr_setup(const Par& q, int ew, const double (&st)[4], Corr& c) {
  if (ew == kNative) return false;
  int eo = ew > -4000 ? ew + q.ic_e + 2 : -4000;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int e = bexp(st[j]);
    if (e > kMaxE + 60) return false;
    // |st 2^t| < 2^(e - 1022 + t); its integer st 2^(t + 4 - eo) must stay below 2^60
    const int need = e - 1022 + q.t[j] - 56;
    if (e >= 64 && need > eo) eo = need;
  }
  if (eo < -900) eo = -900;
  c.eo = eo;
  // W / c in output units: ic 2^(ew + ic_e - 62 - eo), as a 64-bit fraction
  const int r = eo - ew - q.ic_e - 2;
  c.cw = ew > -4000 ? (shr(q.ic, r) + 4) & ~7ull : 0ull;
  // Rounding of the sum, in 2^-32 of an output unit: a truncated product is half a unit low on
  // average, a dropped low product lo lo / 2^64, with the table's mean low word over the chunk (a
  // statistical half instead would leave the chunk's sum, and with it the conserved mass, with a bias of
  // a few hundredths of a unit a point); nothing when all is zero.  A product with a word that is the bias
  // alone is exact: table values that have decayed below 2^-28 of the largest, at half of a chunk's points for
  // small a, would otherwise be made up for too (up to 0.7 of a unit a point).
  uint64_t init = c.cw ? (1ull << 32) + (lo32(c.cw) >> 1) : 0ull;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    // integer = st 2^(t + 4 - eo): to_fixed's shift for x 2^(nb - top) with nb - top = t + 4 - eo
    const int E = 64 + 1022 - (q.t[j] + 4 - eo);
    // whole sixteenths (the bias terms are then whole numbers), the magnitude rounded to nearest: a
    // rounding that is not symmetric in sign would leave a bias
    const uint64_t sb = dbits(st[j]);
    const uint64_t v = bexp(st[j]) >= 64 ? (to_fixed(sb & 0x7fffffffffffffffull, E) + 8) & ~15ull : 0ull;
    c.u[j] = (static_cast<int64_t>(sb) < 0 ? 0ull - v : v) + kCoefBias;
    if (c.u[j] != kCoefBias)
      init += static_cast<uint64_t>(q.trunc_hi[j]) + (hi32(c.u[j]) != hi32(kCoefBias) ? q.trunc_lo[j] : 0u) +
              mad_hi(q.low[j], lo32(c.u[j]), 0u);
  }
  // bias terms that do not depend on k: W's bias times cw; the tables' bias times the states
  uint64_t k0 = c.cw >> 2;  // 2^62 cw / 2^64
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    k0 += static_cast<uint64_t>(static_cast<int64_t>(c.u[j] - kCoefBias) >> 4);
  }
  c.k0 = 0ull - k0;
  c.init = init;
  return true;
}

__host__ __device__ __forceinline__ uint64_t corr_point(const Corr& c, uint64_t W, const uint64_t* t, uint64_t base) {
  uint32_t A = hi32(wmul(lo32(W), hi32(c.cw)) + c.init);
  uint32_t B = mad_hi(hi32(W), lo32(c.cw), 0u);
  uint64_t M = wmul(hi32(W), hi32(c.cw)) + (base + c.k0);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    A = mad_hi(lo32(t[j]), hi32(c.u[j]), A);
    B = mad_hi(hi32(t[j]), lo32(c.u[j]), B);
    M += wmul(hi32(t[j]), hi32(c.u[j]));
  }
  return M + A + B;
}

// x at point k of a chunk in FP64 (the chunk's W at scale mark ew)
__host__ __device__ __forceinline__ double corr_native(const Par& q, int ew, uint64_t W, const uint64_t* t,
                                                       const double (&st)[4]) {
  double x = ew == kNative ? from_bits(W) * (q.inv_c / q.bs)
             : ew > -4000  ? static_cast<double>(static_cast<int64_t>(W - kBias)) * pow2(ew) * q.inv_c
                           : 0.0;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    x = fma(static_cast<double>(static_cast<int64_t>(t[j] - kCoefBias)) * pow2(q.t[j] - 60), st[j], x);
  return x;
}

// ---- host: constants and tables --------------------------------------------------------------------
// Double-double arithmetic, ~2^-104: Knuth's two-sum, Dekker's renormalisation, products' errors by FMA.
struct DD {
  double h, l;
  DD(double a = 0.0, double b = 0.0) : h(a), l(b) {}
};
inline DD dd_norm(double a, double b) {
  const double s = a + b;
  return DD(s, b - (s - a));
}
inline DD operator+(DD a, DD b) {
  const double s = a.h + b.h, t = s - a.h;
  const double e = (a.h - (s - t)) + (b.h - t);
  return dd_norm(s, e + a.l + b.l);
}
inline DD operator-(DD a) { return DD(-a.h, -a.l); }
inline DD operator-(DD a, DD b) { return a + (-b); }
inline DD operator*(DD a, DD b) {
  const double p = a.h * b.h, e = std::fma(a.h, b.h, -p);
  return dd_norm(p, e + (a.h * b.l + a.l * b.h));
}
inline DD operator/(DD a, DD b) {
  const double q0 = a.h / b.h;
  const DD r = a - b * DD(q0);
  const double q1 = r.h / b.h;
  const DD r2 = r - b * DD(q1);
  return dd_norm(q0, q1) + DD(r2.h / b.h);
}
inline DD dd_sqrt(DD a) {
  if (a.h == 0.0) return DD();
  const double x = std::sqrt(a.h);
  const DD r = a - DD(x) * DD(x);
  return dd_norm(x, r.h / (2.0 * x));
}
inline double dd_val(DD a) { return a.h + a.l; }
// nearest integer to v 2^k
inline int64_t dd_int(DD v, int k) {
  const double h = std::ldexp(v.h, k), l = std::ldexp(v.l, k);
  const double r = std::nearbyint(h);
  return static_cast<int64_t>(r) + static_cast<int64_t>(std::nearbyint((h - r) + l));
}
struct M2 {
  DD a, b, c, d;
};
inline M2 mul(const M2& x, const M2& y) {
  return {x.a * y.a + x.b * y.c, x.a * y.b + x.b * y.d, x.c * y.a + x.d * y.c, x.c * y.b + x.d * y.d};
}
inline M2 sub_from_id(const M2& x) { return {DD(1.0) - x.a, -x.b, -x.c, DD(1.0) - x.d}; }
inline M2 add(const M2& x, const M2& y) { return {x.a + y.a, x.b + y.b, x.c + y.c, x.d + y.d}; }
inline M2 inv(const M2& x) {
  const DD det = x.a * x.d - x.b * x.c;
  return {x.d / det, -x.b / det, -x.c / det, x.a / det};
}
inline void put(const M2& x, double* o) {
  o[0] = dd_val(x.a); o[1] = dd_val(x.b); o[2] = dd_val(x.c); o[3] = dd_val(x.d);
}

// Constants and tables of lines of n points in P chunks, for the coefficient a.  tab: m rows; base: m;
// mats: 8 doubles per chunk, A^(m (p + 1)) and (reflected lines) the response of the backward state
// before chunk p to a unit forward state entering the line.  False when the constants leave the
// representable range (a not finite).
inline bool build(int64_t n, int P, double a, bool noflux, Par& q, std::vector<TabRow>& tab,
                  std::vector<uint64_t>& base, std::vector<double>& mats) {
  memset(&q, 0, sizeof q);
  if (!(a >= 0.0) || !std::isfinite(a)) return false;
  q.native = a > 1e24;
  const int m = static_cast<int>(n / P);
  // beyond 1e40 a line of 65536 points or less is its mean to 2^-70, and the constants' last digits would be lost
  // in 1 - A^n
  a = std::min(a, 1e40);
  const DD r = dd_sqrt(DD(1.0) + DD(16.0) * DD(a));
  const DD g = dd_sqrt((DD(1.0) + r) * DD(0.5));
  const DD eta = DD(2.0) / (g * (g + DD(1.0))), eps = DD(2.0) / (g + DD(1.0)), qq = DD(1.0) - eps;
  const DD ic = eta * eta;
  q.eta = dd_val(eta);
  q.eps = dd_val(eps);
  q.inv_c = dd_val(ic);
  q.wide = g.h <= 2.25;
  q.fs = std::ldexp(1.0, std::ilogb(eta.h));
  q.bs = std::ldexp(1.0, std::ilogb(ic.h));
  auto frac = [&](DD v) {  // v 2^64 (or 2^62), a multiple of 4; v <= 1 and < 0.8 when not wide
    const int k = q.wide ? 60 : 62;
    return static_cast<uint64_t>(dd_int(v, k)) << 2;
  };
  q.cn = frac(eta);
  q.ce = frac(eps);
  int e;
  std::frexp(ic.h, &e);  // 1 / c in [2^(e-1), 2^e)
  q.ic = static_cast<uint64_t>(dd_int(ic, 62 - e));
  q.ic_e = e;
  if (q.ic >= (1ull << 62)) q.ic = (1ull << 62) - 1;
  // gains of the zero-state recursion over one chunk
  {
    double Y = 0.0, D = 0.0, gy = 0.0, gd = 0.0;  // y's and D's
    for (int k = 0; k < m; ++k) {
      D = D + ((k == 0 ? 1.0 : 0.0) - std::fma(q.eta, Y, q.eps * D));
      Y += D;
      gy += std::fabs(Y);
      gd += std::fabs(D);
    }
    // W's gain: gy^2 bounds it; short chunks take the exact largest row sum of the two recursions
    // (up to a fifth of the bound), which keeps one or two more bits of W
    double gw = gy * gy, ge = gy * gd;
    if (m <= 256) {
      std::vector<double> rw(m, 0.0), re(m, 0.0), y(m);
      for (int j = 0; j < m; ++j) {
        double Yj = 0.0, Dj = 0.0;
        for (int k = j; k < m; ++k) {
          Dj = Dj + ((k == j ? 1.0 : 0.0) - std::fma(q.eta, Yj, q.eps * Dj));
          Yj += Dj;
          y[k] = Yj;
        }
        double W = 0.0, E = 0.0;
        for (int k = m - 1; k >= 0; --k) {
          E = E + ((k >= j ? y[k] : 0.0) - std::fma(q.eta, W, q.eps * E));
          W += E;
          rw[k] += std::fabs(W);
          re[k] += std::fabs(E);
        }
      }
      gw = *std::max_element(rw.begin(), rw.end());
      ge = *std::max_element(re.begin(), re.end());
    }
    const double G = std::max(gy, gd) * 1.0001, Gw = std::max(gw, 0.5 * ge) * 1.0002;
    q.nb = std::min(61, static_cast<int>(std::floor(62.0 - std::log2(G))));
    q.s2 = std::max(0, static_cast<int>(std::ceil(std::log2(Gw))) + q.nb - 61);
    q.native = q.native || q.nb < 8 || q.s2 > 60;
    q.s2 = std::min(q.s2, 60);
  }
  const uint64_t comp = (static_cast<uint64_t>(lo32(q.cn)) + lo32(q.ce)) >> 1;
  q.init_a = (1ull << 31) + (comp >> 1);
  q.init_b = (1ull << 31) + (comp >> 1);
  q.init_a2 = q.init_a - ((1ull << 31) - ((1ull << 31) >> q.s2));  // not used with wide coefficients
  {
    // the bias's own product, a whole number
    const uint64_t M = (q.cn >> 2) + (q.ce >> 2);
    q.kc = q.wide ? M << 2 : M;
    q.kc2 = q.kc - (kBias >> q.s2);
  }
  const M2 A{DD(1.0) - eta, DD(1.0) - eps, -eta, DD(1.0) - eps};
  // homogeneous responses, per unit of the scaled states
  const DD icf = ic / DD(q.fs), icb = ic / DD(q.bs), bf(q.bs / q.fs);
  std::vector<DD> h[4];
  for (int j = 0; j < 4; ++j) h[j].resize(m);
  M2 Rr;
  DD Rv[2][2];
  for (int j = 0; j < 2; ++j) {
    DD Y = j == 0 ? DD(1.0) : DD(), D = j == 1 ? DD(1.0) : DD();
    for (int k = 0; k < m; ++k) {
      D = D - (eta * Y + eps * D);
      Y = Y + D;
      h[j][k] = Y;
    }
    DD W, E;
    for (int k = m - 1; k >= 0; --k) {
      E = E + h[j][k] - (eta * W + eps * E);
      W = W + E;
      h[j][k] = icf * W;
    }
    Rv[0][j] = bf * W;
    Rv[1][j] = bf * E;
  }
  Rr = {Rv[0][0], Rv[0][1], Rv[1][0], Rv[1][1]};
  for (int j = 0; j < 2; ++j) {
    DD W = j == 0 ? DD(1.0) : DD(), E = j == 1 ? DD(1.0) : DD();
    for (int k = m - 1; k >= 0; --k) {
      E = E - (eta * W + eps * E);
      W = W + E;
      h[2 + j][k] = icb * W;
    }
  }
  tab.assign(m, TabRow{});
  base.assign(m, 0);
  for (int j = 0; j < 4; ++j) {
    double mx = 0.0;
    for (int k = 0; k < m; ++k) mx = std::max(mx, std::fabs(h[j][k].h));
    int t = -900;
    if (mx > 0.0) std::frexp(mx * (1.0 + 0x1p-40), &t);
    t = std::max(t, -900);
    q.t[j] = t;
    uint64_t lows = 0, lo_used = 0, hi_used = 0;
    DD left;  // what rounding the values so far left over, so that their sum is rounded only once
    for (int k = 0; k < m; ++k) {
      const int64_t near = dd_int(h[j][k] + left, 56 - t);
      left = h[j][k] + left - DD(std::ldexp(static_cast<double>(near >> 20), t - 36)) - DD(std::ldexp(static_cast<double>(near & 0xfffff), t - 56));
      const int64_t v = near * 16;  // whole sixteenths of 2^-60
      tab[k].v[j] = static_cast<uint64_t>(v) + kCoefBias;
      base[k] -= tab[k].v[j] >> 4;
      lows += lo32(tab[k].v[j]);
      lo_used += lo32(tab[k].v[j]) != 0;
      hi_used += hi32(tab[k].v[j]) != hi32(kCoefBias);
    }
    q.low[j] = static_cast<uint32_t>(lows / m);
    q.trunc_lo[j] = static_cast<uint32_t>((lo_used << 31) / m);
    q.trunc_hi[j] = static_cast<uint32_t>((hi_used << 31) / m);
  }
  put(Rr, q.R);
  M2 Am{DD(1.0), DD(), DD(), DD(1.0)}, sq = A;
  for (int k = m; k > 0; k >>= 1, sq = mul(sq, sq))
    if (k & 1) Am = mul(Am, sq);
  put(Am, q.M);
  M2 lv = Am;
  q.levels = 0;
  for (int l = 0; l < 6; ++l, lv = mul(lv, lv)) {
    put(lv, q.Ml[l]);
    // |A^k| below 2^-70: what the level would add is below every sum's last bits
    double mx = 0.0;
    for (double v : q.Ml[l]) mx = std::max(mx, std::fabs(v));
    if (mx > 0x1p-70) q.levels = l + 1;
  }
  {
    // the wrapped scan over 2^k >= P chunks counts a chunk twice when P is not a power of two
    double mx = 0.0, v[4];
    M2 full{DD(1.0), DD(), DD(), DD(1.0)}, b = Am;
    for (int k = P; k > 0; k >>= 1, b = mul(b, b))
      if (k & 1) full = mul(full, b);
    put(full, v);
    for (double w : v) mx = std::max(mx, std::fabs(w));
    q.cyclic = !noflux && (P & (P - 1)) == 0 && mx < 0x1p-70;
  }
  mats.assign(static_cast<size_t>(8) * P, 0.0);
  std::vector<M2> pw(P + 1);  // A^(m p)
  pw[0] = {DD(1.0), DD(), DD(), DD(1.0)};
  for (int p = 0; p < P; ++p) {
    pw[p + 1] = mul(pw[p], Am);
    put(pw[p + 1], &mats[8 * p]);
  }
  if (!noflux) {
    put(inv(sub_from_id(pw[P])), q.C);
  } else {
    // mirrored ends: (W, E) after the line = V (y, D) there; (y, D) before it = Q (W, E) at its start
    const DD vs = bf / eta, qs = eta / bf;
    const M2 V{vs, qq / eps * vs, DD(), bf / eps}, Q{qs, -(qq / bf), DD(), eps / bf};
    put(V, q.V);
    M2 N = add(mul(Rr, pw[P - 1]), mul(Am, mul(V, pw[P])));
    for (int p = P - 1;; --p) {
      put(N, &mats[8 * p + 4]);
      if (p == 0) break;
      N = add(mul(Rr, pw[p - 1]), mul(Am, N));
    }
    put(mul(inv(sub_from_id(mul(Q, N))), Q), q.Z);
  }
  return true;
}

// The states entering the chunks of one line on the host: the kernels' scan, in its order.
inline void reduce_host(const Par& q, const std::vector<double>& mats, int P, bool noflux,
                        const std::vector<double>& ends, std::vector<double>& st) {
  std::vector<double> v(2 * P), u(2 * P);
  auto scan = [&](bool fwd) {
    for (int l = 0; (1 << l) < P && l < q.levels; ++l) {
      const int d = 1 << l;
      for (int p = 0; p < P; ++p) {
        int o = fwd ? p - d : p + d;
        if (q.cyclic) o = (o + P) % P;
        if (o >= 0 && o < P)
          mv_add(q.Ml[l], v[2 * o], v[2 * o + 1], v[2 * p], v[2 * p + 1], u[2 * p], u[2 * p + 1]);
        else
          u[2 * p] = v[2 * p], u[2 * p + 1] = v[2 * p + 1];
      }
      v.swap(u);
    }
  };
  st.assign(4 * P, 0.0);
  for (int p = 0; p < P; ++p) v[2 * p] = ends[4 * p], v[2 * p + 1] = ends[4 * p + 1];
  scan(true);
  const std::vector<double> f = v;
  double t0 = 0.0, t1 = 0.0;
  if (!noflux) mv_add(q.C, f[2 * P - 2], f[2 * P - 1], 0.0, 0.0, t0, t1);
  for (int p = 0; p < P; ++p) {
    const int o = p > 0 ? p - 1 : P - 1;
    double y0 = 0.0, y1 = 0.0;
    if (q.cyclic) y0 = f[2 * o], y1 = f[2 * o + 1];
    else if (!noflux) mv_add(&mats[8 * o], t0, t1, f[2 * o], f[2 * o + 1], y0, y1);
    else if (p > 0) y0 = f[2 * o], y1 = f[2 * o + 1];
    st[4 * p] = y0;
    st[4 * p + 1] = y1;
    mv_add(q.R, y0, y1, ends[4 * p + 2], ends[4 * p + 3], v[2 * p], v[2 * p + 1]);
  }
  if (noflux) {
    double w0, w1;
    mv_add(q.V, f[2 * P - 2], f[2 * P - 1], 0.0, 0.0, w0, w1);
    mv_add(q.M, w0, w1, v[2 * P - 2], v[2 * P - 1], v[2 * P - 2], v[2 * P - 1]);
  }
  scan(false);
  double z0, z1;
  mv_add(noflux ? q.Z : q.C, v[0], v[1], 0.0, 0.0, z0, z1);
  for (int p = 0; p < P; ++p) {
    if (q.cyclic) {
      const int o = p + 1 < P ? p + 1 : 0;
      st[4 * p + 2] = v[2 * o];
      st[4 * p + 3] = v[2 * o + 1];
    } else if (!noflux) {
      const int o = p + 1 < P ? p + 1 : 0;
      mv_add(&mats[8 * (P - 1 - o)], z0, z1, v[2 * o], v[2 * o + 1], st[4 * p + 2], st[4 * p + 3]);
    } else {
      if (p > 0) mv_add(&mats[8 * (p - 1)], z0, z1, st[4 * p], st[4 * p + 1], st[4 * p], st[4 * p + 1]);
      else st[0] = z0, st[1] = z1;
      if (p + 1 < P) {
        mv_add(&mats[8 * (p + 1) + 4], z0, z1, v[2 * p + 2], v[2 * p + 3], st[4 * p + 2], st[4 * p + 3]);
      } else {
        double y0, y1;
        mv_add(&mats[8 * (P - 1)], z0, z1, f[2 * P - 2], f[2 * P - 1], y0, y1);
        mv_add(q.V, y0, y1, 0.0, 0.0, st[4 * p + 2], st[4 * p + 3]);
      }
    }
  }
}

// One line on the host, with the kernels' functions in their order.
struct HostAcc {
  uint64_t* p;
  __host__ __device__ void load8(int k, uint64_t (&v)[8]) const { memcpy(v, p + k, 64); }
  __host__ __device__ void store8(int k, const uint64_t (&v)[8]) const { memcpy(p + k, v, 64); }
  __host__ __device__ uint64_t get(int k) const { return p[k]; }
  __host__ __device__ void put(int k, uint64_t v) const { p[k] = v; }
};
inline void solve_host(const Par& q, const std::vector<TabRow>& tab, const std::vector<uint64_t>& base,
                       const std::vector<double>& mats, int64_t n, int P, bool noflux, const double* b, double* x) {
  const int m = static_cast<int>(n / P);
  std::vector<uint64_t> w(n);
  std::vector<double> ends(4 * P), st;
  std::vector<int> ew(P);
  memcpy(w.data(), b, 8 * n);
  for (int p = 0; p < P; ++p) {
    HostAcc s{w.data() + static_cast<size_t>(p) * m};
    double e[4];
    ew[p] = local_solve(q, s, s, m, e);
    for (int j = 0; j < 4; ++j) ends[4 * p + j] = e[j];
  }
  reduce_host(q, mats, P, noflux, ends, st);
  for (int p = 0; p < P; ++p) {
    double s4[4] = {st[4 * p], st[4 * p + 1], st[4 * p + 2], st[4 * p + 3]};
    Corr c;
    const bool fixed = corr_setup(q, ew[p], s4, c);
    for (int k = 0; k < m; ++k) {
      const uint64_t W = w[static_cast<size_t>(p) * m + k];
      x[static_cast<size_t>(p) * m + k] = fixed ? from_fixed(corr_point(c, W, tab[k].v, base[k]), c.eo)
                                                : corr_native(q, ew[p], W, tab[k].v, s4);
    }
  }
}

}  // namespace pn
}  // namespace cs
