// Cahn-Hilliard ADI time step with periodic boundaries (Sec. 5.1 of arXiv:1902.09931).
//
//   Cbar = 2 C^n - C^{n-1}
//   RHS  = -(2/3)(C^n - C^{n-1}) - (2/3) D gamma dt lap4(Cbar) + (2/3) D dt lap2(C^3 - C)^n
//   L_x w = RHS,   L_y v = w,   C^{n+1} = Cbar + v,   L = I + a P,  a = (2/3) D gamma dt / h^4
//
// lap2 is the 5-point Laplacian of Eq. 5a and lap4 = dxxxx + 2 dxxyy + dyyyy (Eq. 5b, Fig. 1),
// which on the periodic grid is exactly lap2 applied twice.  The right-hand side is therefore
// evaluated in the factored form
//   Z   = (2/3) D dt / h^2 * N - a * (sum of 4 neighbours of Cbar - 4 Cbar)
//   RHS = -(2/3)(C^n - C^{n-1}) + (sum of 4 neighbours of Z - 4 Z)
// which needs 16 instead of 24 FP64 operations per point (FP64 is the bound on GB300); the two
// Laplacians are exact integer-digit sums, each scaled by one FP64 FMA (the first carrying -a), which
// leaves about 8.6.  FP32 storage evaluates the right-hand side the same way, on exactly widened
// values: its terms reach ~64 a |Cbar| and the solves cancel them back down to |C|, so FP32
// arithmetic there would lose every digit of C at n = 4096 (a = 1.8e5).
//
// Line solves (the paper uses cuPentBatch with the periodic corners treated as in Navon's
// PENT): cs_penta.cuh's factored recursions in 64-bit fixed point, every line cut into P chunks of
// m = n / P points, one thread per (line, chunk).  Two launches a step, one along the rows and one along
// the columns with the update fused; each holds its lines in shared memory, so the field is read
// once and written once.  4096^2, FP64 storage, periodic: rows 166 us (DRAM floor 39 us, bound by the
// integer pipes), columns 232 us (floor 59 us), the step
// 0.60 ms (0.86 ms with FP64 recursions); 1024^2 65 us (110).
//
// No-flux boundaries (cs_ch_desc.boundary = CS_CH_NOFLUX): the same step on a cell-centred
// grid whose stencils read ghost cells by even reflection.  Reflection commutes with the
// 5-point Laplacian, so the factored right-hand side holds unchanged -- only the tile loader
// mirrors indices instead of wrapping them.  The line operator is I + a D4 with the reflected fourth
// difference (first rows (1+2a, -3a, a), (-3a, 1+6a, -4a, a)): the recursions are the same, only the
// states entering the first and last chunks follow from the mirror conditions instead of the wrap.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <type_traits>
#include <vector>

#include <cooperative_groups.h>

#include "cs_digits.cuh"
#include "cs_internal.h"
#include "cs_penta.cuh"

namespace cs {

// The line solver of a plan (cs_penta.cuh): constants, device tables (mats, then the table rows, then
// the bias terms, in one allocation), and the scratch of the kernels that work from global memory (end
// values, states, scale marks), allocated only for plans that run them.
struct Lines {
  pn::Par par;
  double* tables;
  double* scratch;
  int P, m;
};

struct CHPlan {
  int64_t n;
  int storage;
  double D, gamma, dt, h, a, alpha;
  int P, m;
  void* field[3];
  int iprev, icur, inext;
  int64_t steps;
  double* A;         // n*n scratch (RHS, then w)
  double* B;         // n*n scratch (local solutions of lines too long for shared memory; coarsening)
  Lines lines;       // the line solver's constants, tables and (long lines only) scratch
  double* partials;  // 2 per RHS block
  double* inv;       // 2 per step (device)
  int64_t inv_cap;
  int rhs_blocks;
  cudaGraphExec_t graph3[3];  // three steps (one buffer rotation) per starting rotation phase
  int graph_kernels;
  double* diag;  // coarsening measures: n/2 twiddles (re, im), 2 n partial sums, 4 results
  int noflux;    // CS_CH_NOFLUX: reflected ghost cells, non-cyclic line solves
};

void drop_graphs(CHPlan* p);

namespace {

constexpr int kTX = 64, kTY = 32, kThreads = 256, kSolveThreads = 32;
constexpr int kU = 8;  // line elements per register batch in the solves

// ---- exact conversions on the integer pipe (f32 <-> f64 conversion runs on the FP64 pipe) ----
__device__ __forceinline__ double widen(float f) {
  const uint32_t b = __float_as_uint(f);
  const uint32_t e = (b >> 23) & 0xffu;
  if (e == 0u || e == 0xffu) {
    if ((b & 0x7fffffffu) == 0u) return __longlong_as_double(static_cast<long long>(b & 0x80000000u) << 32);
    return static_cast<double>(f);  // subnormal, inf, nan: rare
  }
  const uint64_t d = (static_cast<uint64_t>(b & 0x80000000u) << 32) |
                     (static_cast<uint64_t>(e + 896u) << 52) |
                     (static_cast<uint64_t>(b & 0x7fffffu) << 29);
  return __longlong_as_double(static_cast<long long>(d));
}
__device__ __forceinline__ double widen(double d) { return d; }

__device__ __forceinline__ float narrow_rn(double x) {
  const uint64_t b = static_cast<uint64_t>(__double_as_longlong(x));
  const int e = static_cast<int>((b >> 52) & 0x7ffu) - 1023 + 127;
  if (e <= 0 || e >= 255) {
    if ((b << 1) == 0) return __uint_as_float(static_cast<uint32_t>(b >> 32));  // +-0
    return __double2float_rn(x);  // subnormal result, overflow, inf, nan: rare
  }
  const uint32_t sign = static_cast<uint32_t>(b >> 32) & 0x80000000u;
  const uint64_t mant = b & 0xFFFFFFFFFFFFFull;
  const uint32_t m23 = static_cast<uint32_t>(mant >> 29);
  const uint32_t rem = static_cast<uint32_t>(mant & 0x1FFFFFFFu);
  uint32_t r = sign | (static_cast<uint32_t>(e) << 23) | m23;
  if (rem > 0x10000000u || (rem == 0x10000000u && (m23 & 1u))) r += 1u;  // ties to even
  return __uint_as_float(r);
}

// ---- the cubic term of Z on the Laplacian's digit grid ----------------------------------------
// Z = alpha N - a Lap(Cbar), N = u^3 - u (u = C^n).  Lap(Cbar) is an exact digit sum T on the grid
// 2^(G-56) of Cbar's tile, combined as (T' + Q) c 2^(G-48) with T' = round(T / 2^8) and c = -a
// rounded to 51 bits (ixi_combine<28>).  N joins it as the integer Q = round(alpha N / (c 2^(G-48))),
// formed in double-float arithmetic on the FP32 pipe, two points per packed instruction; Z then
// costs the one FP64 FMA of the combination instead of four FP64 operations.  Q is rounded to the
// grid unit c 2^(G-48) that T' already has, so Z's error stays of the size of the Laplacian's own
// rounding.  Used where alpha / |c| <= 2^-6 (the host passes a zero inverse otherwise), which keeps
// the double-float error of Q (<= 2^-46 |alpha N| plus 2^-47 |u| |3u^2 - 1| alpha / |c| in grid
// units) below a tenth of a unit; points outside the ranges below take the FP64 formula.
struct CubicInv { float hi, lo; };  // alpha / c as a float pair, or zero: the FP64 formula

inline CubicInv cubic_inv(double alpha, double c) {
  const double r = alpha / c;
  if (!(std::fabs(r) <= 0.015625) || r == 0.0) return {0.0f, 0.0f};
  const float hi = static_cast<float>(r);
  return {hi, static_cast<float>(r - static_cast<double>(hi))};
}

// (alpha / c) 2^(48 - G) as a float pair, by exponent arithmetic on the host's pair; false when
// the inverse is zero or the scaled pair would leave the normal float range.
__device__ __forceinline__ bool cubic_scaled(CubicInv inv, int tile_e, float& ih, float& il) {
  const int sh = 1070 - tile_e;  // 48 - G, G = tile_e - 1022
  const int eh = static_cast<int>((__float_as_uint(inv.hi) >> 23) & 0xffu) + sh;
  if (inv.hi == 0.0f || eh < 25 || eh > 254) return false;
  ih = __uint_as_float(__float_as_uint(inv.hi) + (static_cast<uint32_t>(sh) << 23));
  const int el = static_cast<int>((__float_as_uint(inv.lo) >> 23) & 0xffu) + sh;
  il = (inv.lo == 0.0f || el < 1) ? 0.0f : __uint_as_float(__float_as_uint(inv.lo) + (static_cast<uint32_t>(sh) << 23));
  return true;
}

// u as the float pair h + l with |u - h - l| < 2^-47 |u|, by integer operations alone: h holds u's
// sign, exponent and leading 24 significand bits, l the next 24 bits.  Valid for biased exponents
// e in [944, 1150]; e = 0 (zero or subnormal) gives h = l = 0.
__device__ __forceinline__ void split_hl(double u, float& h, float& l) {
  const uint32_t hw = static_cast<uint32_t>(__double2hiint(u)), lw = static_cast<uint32_t>(__double2loint(u));
  // hw << 3 | lw >> 29 puts the exponent's low 8 bits over the top 23 significand bits; with the
  // exponent's bit 7 flipped first those 8 bits read e - 896, the float exponent (e in [897, 1150])
  const uint32_t top = __funnelshift_l(lw, hw ^ 0x08000000u, 3);
  const uint32_t hb = (top & 0x7fffffffu) | (hw & 0x80000000u);
  // the next 24 bits as an exact integer times 2^(e - 1070), with u's sign: float exponent e - 943
  const float x = __uint2float_rn((lw >> 5) & 0xffffffu);
  const float sc = __uint_as_float((hb & 0xff800000u) - (47u << 23));
  const bool zero = (hw & 0x7ff00000u) == 0u;
  h = zero ? 0.0f : __uint_as_float(hb);
  l = zero ? 0.0f : __fmul_rn(x, sc);
}

__device__ __forceinline__ float2 f2s(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, f2s(-1.0f), a); }

// Q for two points u = h + l (packed lanes), returned as qa 2^20 + qb, the split ixi_combine<28>
// takes, with qh (|qh| < 2^43 is required; the caller checks it).  Steps, all error-free apart from
// the dropped l^2 and a l terms (2^-48 relative) and the roundings of the small parts:
//   u^2 = A + a2:   nA = -h h rounded, a2 = (h h + nA) + 2 h l
//   u^3 = s3 + b:   ns3 = nA h rounded (= -s3), b = (A h - s3) + A l + a2 h
//   -N = u - u^3 = (ns3 + h) + (l - b) = S + lo (TwoSum of ns3 and h)
//   R = -N (alpha / c) 2^(48 - G) = qh + ql (the product's error by FMA, renormalised by Fast2Sum)
// and Q = -round(R) in two FP32 rounding shifts: 1.5 2^44 takes qh to k 2^21 (k in the low
// mantissa bits), 1.5 2^23 rounds the rest (qh - k 2^21 + ql, |rest| < 2^21) to k2; Q = -(k 2^21 + k2).
__device__ __forceinline__ void cubic_q2(float2 h, float2 l, float ih, float il, int2& qa, int2& qb, float2& qh) {
  const float2 nh = __fmul2_rn(h, f2s(-1.0f)), nl = __fmul2_rn(l, f2s(-1.0f));
  const float2 nA = __fmul2_rn(nh, h);
  const float2 a2 = __ffma2_rn(__fadd2_rn(h, h), l, __ffma2_rn(h, h, nA));
  const float2 ns3 = __fmul2_rn(nA, h);
  float2 b = __ffma2_rn(nA, nh, ns3);
  b = __ffma2_rn(nA, nl, b);
  b = __ffma2_rn(a2, h, b);
  const float2 S = __fadd2_rn(ns3, h);
  const float2 bb = sub2(S, ns3);
  const float2 t = __fadd2_rn(sub2(ns3, sub2(S, bb)), sub2(h, bb));
  const float2 lo = __fadd2_rn(sub2(t, b), l);
  const float2 np = __fmul2_rn(S, f2s(-ih));
  float2 pl = __ffma2_rn(S, f2s(ih), np);
  pl = __ffma2_rn(lo, f2s(ih), pl);
  pl = __ffma2_rn(S, f2s(il), pl);
  qh = sub2(pl, np);
  const float2 ql = sub2(pl, __fadd2_rn(qh, np));
  constexpr float M1 = 26388279066624.0f, M2 = 12582912.0f;  // 1.5 2^44, 1.5 2^23
  const float2 t1 = __fadd2_rn(qh, f2s(M1));
  const float2 rest = __fadd2_rn(sub2(qh, sub2(t1, f2s(M1))), ql);
  const float2 t2 = __fadd2_rn(rest, f2s(M2));
  qa = make_int2(2 * static_cast<int>(__float_as_uint(M1) - __float_as_uint(t1.x)),
                 2 * static_cast<int>(__float_as_uint(M1) - __float_as_uint(t1.y)));
  qb = make_int2(static_cast<int>(__float_as_uint(M2) - __float_as_uint(t2.x)),
                 static_cast<int>(__float_as_uint(M2) - __float_as_uint(t2.y)));
}

// Whether a point may take the digit form: u zero or with biased exponent in [944, tile_e + 1]
// (|u| < 2^(G+1), which bounds the double-float error of Q), |qh| < 2^43 (the rounding shifts'
// range; false for inf and nan), and the Laplacian's high digit sum |S0| <= 2^31 - 2^24, so that
// |T' + Q| < 2^51 as the combination requires.
__device__ __forceinline__ bool cubic_ok(double u, int tile_e, float qh, int s0) {
  const int e = static_cast<int>((static_cast<uint32_t>(__double2hiint(u)) >> 20) & 0x7ffu);
  return (e == 0 || (e >= 944 && e <= tile_e + 1)) && fabsf(qh) < 8796093022208.0f &&
         abs(s0) <= 2147483647 - 16777215;
}

// 2^k as a double (k in the normal range), by its bit pattern
__device__ __forceinline__ double pow2d(int k) { return __longlong_as_double(static_cast<long long>(k + 1023) << 52); }

// a 128-bit integer as a double, within 2^-52 of its value: magnitude in two 64-bit halves
__device__ __forceinline__ double i128_to_double(__int128 v) {
  const bool neg = v < 0;
  const unsigned __int128 a = neg ? static_cast<unsigned __int128>(-v) : static_cast<unsigned __int128>(v);
  const double r = fma(__ull2double_rn(static_cast<unsigned long long>(a >> 64)), 18446744073709551616.0,
                       __ull2double_rn(static_cast<unsigned long long>(a)));
  return neg ? -r : r;
}

__device__ __forceinline__ int wrapn(int64_t k, int64_t n) {
  return static_cast<int>(k < 0 ? k + n : (k >= n ? k - n : k));
}
// even reflection about the boundary: -1 -> 0, -2 -> 1, n -> n - 1, n + 1 -> n - 2
__device__ __forceinline__ int mirrorn(int64_t k, int64_t n) {
  return static_cast<int>(k < 0 ? -1 - k : (k >= n ? 2 * n - 1 - k : k));
}
// 128-bit shuffle (two 64-bit halves)
__device__ __forceinline__ __int128 shfl_down_i128(__int128 v, int off) {
  const unsigned long long lo = __shfl_down_sync(0xffffffffu, static_cast<unsigned long long>(v), off);
  const long long hi = __shfl_down_sync(0xffffffffu, static_cast<long long>(v >> 64), off);
  return static_cast<__int128>(hi) * (static_cast<__int128>(1) << 64) + static_cast<__int128>(lo);
}

// The block's exact integer invariant sums (mass digits S0, S1; sum U L; sum W^2, see k_ch_rhs),
// reduced in integers over the block (every total stays below 2^127), then converted once to
// FP64 by thread 0: out2 = (sum C, sum energy density) of the block.
__device__ __forceinline__ void block_reduce_int(long long s0, long long s1, __int128 sg, __int128 sw, int G,
                                                 double half_gamma_over_h2, double* out2) {
  __shared__ long long rs[2][kThreads / 32];
  __shared__ __int128 rq[2][kThreads / 32];
  for (int off = 16; off > 0; off >>= 1) {
    s0 += __shfl_down_sync(0xffffffffu, s0, off);
    s1 += __shfl_down_sync(0xffffffffu, s1, off);
    sg += shfl_down_i128(sg, off);
    sw += shfl_down_i128(sw, off);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) { rs[0][warp] = s0; rs[1][warp] = s1; rq[0][warp] = sg; rq[1][warp] = sw; }
  __syncthreads();
  if (threadIdx.x == 0) {
    long long a = 0, b = 0;
    __int128 g = 0, w = 0;
    for (int k = 0; k < kThreads / 32; ++k) { a += rs[0][k]; b += rs[1][k]; g += rq[0][k]; w += rq[1][k]; }
    out2[0] = fma(static_cast<double>(a), 268435456.0, static_cast<double>(b)) * pow2d(G - 56);
    const double ew = i128_to_double(w) * pow2d(4 * G - 102);
    const double eg = i128_to_double(g) * pow2d(2 * G - 112);
    out2[1] = fma(0.25, ew, -half_gamma_over_h2 * eg);
  }
}

template <typename T>
__device__ __forceinline__ void block_reduce2(double m, double e, double* out2) {
  __shared__ double red[2][kThreads / 32];
  for (int off = 16; off > 0; off >>= 1) {
    m += __shfl_down_sync(0xffffffffu, m, off);
    e += __shfl_down_sync(0xffffffffu, e, off);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) { red[0][warp] = m; red[1][warp] = e; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double sm = 0.0, se = 0.0;
    for (int w = 0; w < kThreads / 32; ++w) { sm += red[0][w]; se += red[1][w]; }
    out2[0] = sm;
    out2[1] = se;
  }
}

// RHS of the x-sweep and, when partials != nullptr, the per-block FP64 sums of C and of the
// free-energy density of C^n.  rhs == nullptr computes the sums only.  The tile is staged in FP64
// whatever the storage type T (FP32 values widen exactly): the right-hand side carries terms of
// size ~64 a |Cbar| (a = 1.8e5 at n = 4096) that the solves cancel back down to |C|, so it needs
// FP64 precision; evaluated in FP32 it loses all of C's digits at the large grids.  The one
// exception: with FP32 storage Cbar = 2 C^n - C^{n-1} is formed in FP32 (one rounding) exactly as
// the update forms it, then widened.  Both uses of Cbar then agree, so the step is the scheme
// applied to that Cbar, whose rounding reaches C^{n+1} at most undamped (it is of the size of the
// stored result's own rounding); everything after it is FP64.  At least 5 CTAs per SM (the two
// staged tiles' 39 KB of shared memory allow 5): 48 registers, no spills.
template <typename T>
__global__ void __launch_bounds__(kThreads, 5)
    k_ch_rhs(const T* __restrict__ cur, const T* __restrict__ prev, double* __restrict__ rhs, int64_t n,
             double alpha, double a, double half_gamma_over_h2, double* __restrict__ partials, int noflux,
             double am51, CubicInv cinv, int band, T* __restrict__ cbar_out) {
  constexpr int HR = kTY + 4, HC = kTX + 4;  // halo-2 tiles
  constexpr int ZR = kTY + 2, ZC = kTX + 2;  // halo-1 tile
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* sc = reinterpret_cast<double*>(smem_raw);  // C^n
  double* sb = sc + HR * HC;                         // Cbar, then Z (halo-1 tile) once Cbar is used up
  const int64_t x0 = static_cast<int64_t>(blockIdx.x) * kTX;
  const int64_t y0 = static_cast<int64_t>(blockIdx.y) * kTY;
  // band != 0: cur and prev are row bands padded with the 2 rows above and the 2 rows below (the
  // neighbours' rows, exchanged by the caller, or at a no-flux edge of the grid the band's own rows
  // mirrored); output row r of the band is padded row r + 2
  const uintptr_t addr_bits = reinterpret_cast<uintptr_t>(cur) | reinterpret_cast<uintptr_t>(prev) |
                              reinterpret_cast<uintptr_t>(cbar_out);
  const bool inner = x0 >= 2 && x0 + kTX + 2 <= n && (band || (y0 >= 2 && y0 + kTY + 2 <= n)) &&
                     (addr_bits & (2 * sizeof(T) - 1)) == 0;
  if (inner) {
    // a tile whose halo lies inside the grid (or inside the padded band): no wrap or mirror, two
    // adjacent values per load and store (x0 - 2 and n are even; 16 bytes for FP64 storage, 8 for
    // FP32), a fixed trip count so that the loads of several pairs are in flight together
    constexpr int HP = HC / 2, NPAIR = HR * HP, IT = (NPAIR + kThreads - 1) / kThreads;
#pragma unroll
    for (int k = 0; k < IT; ++k) {
      const int idx = threadIdx.x + k * kThreads;
      if (k + 1 < IT || idx < NPAIR) {
        const int r = idx / HP, cp = idx - r * HP;
        const int64_t gy = y0 - 2 + r, gx = x0 - 2 + 2 * cp;
        const int64_t off = (band ? gy + 2 : gy) * n + gx;
        const bool own = cbar_out && r >= 2 && r < kTY + 2 && cp >= 1 && cp < HP - 1;
        const int i0 = r * HC + 2 * cp;
        if constexpr (sizeof(T) == 4) {
          const float2 cf = *reinterpret_cast<const float2*>(cur + off);
          const float2 pf = *reinterpret_cast<const float2*>(prev + off);
          const float2 cb = make_float2(fmaf(2.0f, cf.x, -pf.x), fmaf(2.0f, cf.y, -pf.y));
          *reinterpret_cast<double2*>(sc + i0) = make_double2(widen(cf.x), widen(cf.y));
          *reinterpret_cast<double2*>(sb + i0) = make_double2(widen(cb.x), widen(cb.y));
          if (own) *reinterpret_cast<float2*>(cbar_out + gy * n + gx) = cb;
        } else {
          const double2 cd = *reinterpret_cast<const double2*>(cur + off);
          const double2 pd = *reinterpret_cast<const double2*>(prev + off);
          const double2 cb = make_double2(fma(2.0, cd.x, -pd.x), fma(2.0, cd.y, -pd.y));
          *reinterpret_cast<double2*>(sc + i0) = cd;
          *reinterpret_cast<double2*>(sb + i0) = cb;
          if (own) *reinterpret_cast<double2*>(cbar_out + gy * n + gx) = cb;
        }
      }
    }
  }
  for (int idx = inner ? HR * HC : threadIdx.x; idx < HR * HC; idx += kThreads) {
    const int r = idx / HC, c = idx - r * HC;
    const int64_t gy = y0 - 2 + r, gx = x0 - 2 + c;
    const int64_t off = band      ? (gy + 2) * n + (noflux ? mirrorn(gx, n) : wrapn(gx, n))
                        : noflux  ? static_cast<int64_t>(mirrorn(gy, n)) * n + mirrorn(gx, n)
                                  : static_cast<int64_t>(wrapn(gy, n)) * n + wrapn(gx, n);
    const double cv = widen(cur[off]);
    sc[idx] = cv;
    // cbar_out (the step's C^{n+1} buffer, non-null for the full-grid step): the tile's own Cbar,
    // which the fused update then reads instead of forming it again from C^n and C^{n-1}
    const bool own = cbar_out && r >= 2 && r < kTY + 2 && c >= 2 && c < kTX + 2;
    if constexpr (sizeof(T) == 4) {
      const float cb = fmaf(2.0f, cur[off], -prev[off]);  // as the FP32 update forms Cbar
      sb[idx] = widen(cb);
      if (own) cbar_out[gy * n + gx] = cb;
    } else {
      const double cb = fma(2.0, cv, -prev[off]);  // one FP64 instruction (2 cv - p as two adds is two)
      sb[idx] = cb;
      if (own) cbar_out[gy * n + gx] = cb;
    }
  }
  __syncthreads();
  __shared__ __align__(16) unsigned s_red[kThreads / 32];
  auto lap5 = [&](const double* t, int i, int pitch) {
    return (t[i - pitch] + t[i + pitch]) + (t[i - 1] + t[i + 1]) - 4.0 * t[i];
  };
  // digit sums of the 5-point Laplacian at i of a split tile (int2 digits over t's slots)
  auto lap5_digits = [&](const double* t, int i, int pitch, int& q0, int& q1) {
    const int2* d = reinterpret_cast<const int2*>(t);
    const int2 u = d[i - pitch], v = d[i + pitch], w = d[i - 1], x = d[i + 1], c = d[i];
    q0 = (u.x + v.x) + (w.x + x.x) - 4 * c.x;
    q1 = (u.y + v.y) + (w.y + x.y) - 4 * c.y;
  };
  if (rhs) {
    // Both 5-point Laplacians as exact integer-digit sums (weights 1, 1, 1, 1, -4; 28-bit digits, which
    // hold every bit of a value within a factor 8 of its tile's largest, so neighbouring tiles,
    // which evaluate Z on each other's border, agree on it to 2^-56 of the tile's scale and the sum
    // of the Laplacian over the grid stays zero to that level: mass is conserved), each scaled with
    // one FP64 FMA; the first one's scaling carries -a, and the cubic term N joins its digit sum
    // as an integer (cubic_q2), so the FP64 pipe keeps only Cbar, Z, the second scaling,
    // C^n - C^{n-1} and the final combination (5.3 FP64 operations per point).  A tile whose values
    // leave the digit range takes the FP64 formula for that Laplacian; a warp with a point outside
    // cubic_ok's ranges forms N in FP64.
    // the one-FMA scaling of a digit sum by m 2^(G - 56) (ixi_consts); false: the FP64 formula
    double* cb = sb;
    double* zt = sb;  // Z takes Cbar's place (held in registers until every thread has read Cbar)
    const double* cn = sc;
    {
      const int te = static_cast<int>(ixd::ix_tile_max_hi<kThreads, HR * HC>(cb, s_red) >> 20);
      uint32_t w[4];
      const bool dig = ixd::ixi_consts<28>(am51, -1.5 * am51, te, w);  // uniform over the block
      float ih = 0.0f, il = 0.0f;
      const bool cub = dig && te != 0 && cubic_scaled(cinv, te, ih, il);  // uniform too
      if (dig) {
        ixd::ixi_split_tile<kThreads, HR * HC, 28>(cb, te);
        __syncthreads();
      }
      constexpr int NZ = (ZR * ZC + kThreads - 1) / kThreads;
      double zv[NZ];
      // Z point k of this thread: the Laplacian's digit sums and u (a point past the tile reads
      // the first one; its result is not stored)
      auto zpoint = [&](int k, int& q0, int& q1, double& u) {
        int idx = threadIdx.x + k * kThreads;
        if (idx >= ZR * ZC) idx = 0;
        const int r = idx / ZC, c = idx - r * ZC;
        const int hidx = (r + 1) * HC + (c + 1);
        lap5_digits(cb, hidx, HC, q0, q1);
        u = cn[hidx];
      };
      if (cub) {
#pragma unroll
        for (int k = 0; k < NZ; k += 2) {  // two points per packed cubic term
          const int k1 = k + 1 < NZ ? k + 1 : k;
          int a0, a1, b0, b1;
          double u0, u1;
          zpoint(k, a0, a1, u0);
          zpoint(k1, b0, b1, u1);
          float h0, l0, h1, l1;
          split_hl(u0, h0, l0);
          split_hl(u1, h1, l1);
          int2 qa, qb;
          float2 qh;
          cubic_q2(make_float2(h0, h1), make_float2(l0, l1), ih, il, qa, qb, qh);
          const bool ok = cubic_ok(u0, te, qh.x, a0) && cubic_ok(u1, te, qh.y, b0);
          double z0, z1;
          if (__all_sync(0xffffffffu, ok)) {
            z0 = ixd::ixi_combine<28>(a0, a1, w, qa.x, qb.x);
            z1 = ixd::ixi_combine<28>(b0, b1, w, qa.y, qb.y);
          } else {
            z0 = fma(alpha, fma(u0 * u0, u0, -u0), ixd::ixi_combine<28>(a0, a1, w));
            z1 = fma(alpha, fma(u1 * u1, u1, -u1), ixd::ixi_combine<28>(b0, b1, w));
          }
          zv[k] = z0;
          if (k + 1 < NZ) zv[k + 1] = z1;
        }
      } else {
#pragma unroll
        for (int k = 0; k < NZ; ++k) {
          const int idx = threadIdx.x + k * kThreads;
          if (k + 1 < NZ || idx < ZR * ZC) {
            const int r = idx / ZC, c = idx - r * ZC;
            const int hidx = (r + 1) * HC + (c + 1);
            double lap_a;  // -a * Laplacian(Cbar)
            if (dig) {
              int q0, q1;
              lap5_digits(cb, hidx, HC, q0, q1);
              lap_a = ixd::ixi_combine<28>(q0, q1, w);
            } else {
              lap_a = -a * lap5(cb, hidx, HC);
            }
            const double u = cn[hidx];
            zv[k] = fma(alpha, fma(u * u, u, -u), lap_a);
          }
        }
      }
      __syncthreads();  // every thread is done with Cbar
#pragma unroll
      for (int k = 0; k < NZ; ++k) {
        const int idx = threadIdx.x + k * kThreads;
        if (k + 1 < NZ || idx < ZR * ZC) zt[idx] = zv[k];
      }
      __syncthreads();
    }
    {
      const int te = static_cast<int>(ixd::ix_tile_max_hi<kThreads, ZR * ZC>(zt, s_red) >> 20);
      uint32_t w[4];
      const bool dig = ixd::ixi_consts<28>(1.0, -1.5, te, w);
      if (dig) {
        ixd::ixi_split_tile<kThreads, ZR * ZC, 28>(zt, te);
        __syncthreads();
      }
      for (int idx = threadIdx.x; idx < kTY * kTX; idx += kThreads) {
        const int r = idx / kTX, c = idx - r * kTX;
        const int zidx = (r + 1) * ZC + (c + 1);
        const int hidx = (r + 2) * HC + (c + 2);
        double lap_z;
        if (dig) {
          int q0, q1;
          lap5_digits(zt, zidx, ZC, q0, q1);
          lap_z = ixd::ixi_combine<28>(q0, q1, w);
        } else {
          lap_z = lap5(zt, zidx, ZC);
        }
        const int64_t o = (y0 + r) * n + x0 + c;
        const double diff = cn[hidx] - widen(prev[band ? o + 2 * n : o]);  // C^n - C^{n-1}
        rhs[o] = fma(-2.0 / 3.0, diff, lap_z);
      }
    }
  }
  if (partials) {
    // Mass sum C and free-energy density sum (1/4)(C^2 - 1)^2 + (gamma / 2h^2)(|D+x C|^2 + |D+y C|^2)
    // (Eq. 1 with forward differences).  The gradient part is summed by parts: over the periodic
    // grid, and with the even reflection of the no-flux boundary, the sum of the squared forward
    // differences equals -sum C Lap5(C) (Lap5 the unscaled 5-point Laplacian, reading the staged
    // halo).  Lap5(C) is an exact digit sum scaled by one FP64 FMA, so a point costs 5 FP64
    // operations instead of 9; only the grid total (the sum over all blocks, or over all bands
    // with their halos) equals the forward-difference sum, not each block's share.
    __syncthreads();  // sb (Cbar, then Z) is no longer read: it takes C's digits
    const int te = static_cast<int>(ixd::ix_tile_max_hi<kThreads, HR * HC>(sc, s_red) >> 20);
    uint32_t w4[4];
    const bool dig = ixd::ixi_consts<28>(1.0, -1.5, te, w4);  // uniform over the block
    if (dig) {
      constexpr int NP = HR * HC / 2;
      const double2* q = reinterpret_cast<const double2*>(sc);
      int4* qi = reinterpret_cast<int4*>(sb);
      for (int k = threadIdx.x; k < NP; k += kThreads) {
        const double2 v = q[k];
        const int2 a0 = ixd::ixi_split<28>(v.x, te), a1 = ixd::ixi_split<28>(v.y, te);
        qi[k] = make_int4(a0.x, a0.y, a1.x, a1.y);
      }
      __syncthreads();
    }
    double* out2 = partials + 2 * (static_cast<int64_t>(blockIdx.y) * gridDim.x + blockIdx.x);
    const int G = te - 1022;  // the tile's values lie below 2^G
    if (dig && G >= -3 && G <= 3) {
      // Each thread's share in exact integer arithmetic on the digit grid: u = U 2^(G-56) with
      // U = d0 2^28 + d1 (every bit of a value within a factor 8 of the tile's largest), and
      // Lap5(u) = L 2^(G-56) with L = q0 2^28 + q1 the exact digit sums.  Per point, only 32 x 32
      // -> 64-bit multiply-adds into 64-bit sums:
      //   mass      sum d0, sum d1;
      //   U L       sum d0 q0, sum (d0 q1 + d1 q0), sum d1 q1;
      //   u^2 - 1   W = round((U^2 - 2^(112-2G)) / 2^61) (units 2^(2G-51), |W| <= 2^57 + 1), from
      //             A = d0^2 - 2^(56-2G) and B = 2 d0 d1 + floor(d1^2 / 2^28) as
      //             (A >> 5) + ((A mod 32) 2^28 + B + 2^32) >> 33 (d1^2's dropped bits are below
      //             2^-33 of W's unit);
      //   W^2       with W = Wh 2^29 + Wl: sum Wh^2, sum Wh Wl, sum Wl^2.
      // Every sum of the thread's 8 points stays below 2^63; each is joined once in 128 bits, the
      // block reduces them in integers, and thread 0 converts the block's totals to FP64.  No FP64
      // operation per point or per thread (the formula below takes 5 per point, and its FP64
      // shuffle reduction 10 per thread).
      int s0 = 0, s1 = 0;
      long long g2 = 0, g1 = 0, g0 = 0, w2 = 0, w1 = 0, w0 = 0;
      const long long K56 = 1ll << (56 - 2 * G);
      const int2* dg = reinterpret_cast<const int2*>(sb);
      for (int idx = threadIdx.x; idx < kTY * kTX; idx += kThreads) {
        const int r = idx / kTX, c = idx - r * kTX;
        const int hidx = (r + 2) * HC + (c + 2);
        const int2 d = dg[hidx];
        int q0, q1;
        lap5_digits(sb, hidx, HC, q0, q1);
        s0 += d.x;
        s1 += d.y;
        g2 += static_cast<long long>(d.x) * q0;
        g1 += static_cast<long long>(d.x) * q1 + static_cast<long long>(d.y) * q0;
        g0 += static_cast<long long>(d.y) * q1;
        const long long A = static_cast<long long>(d.x) * d.x - K56;
        const long long B = static_cast<long long>(d.x) * (2 * d.y) +
                            static_cast<long long>(static_cast<unsigned long long>(static_cast<unsigned>(d.y)) * static_cast<unsigned>(d.y) >> 28);
        const long long W = (A >> 5) + ((((A & 31) << 28) + B + (1ll << 32)) >> 33);
        const int wh = static_cast<int>(W >> 29), wl = static_cast<int>(W & ((1ll << 29) - 1));
        w2 += static_cast<long long>(wh) * wh;
        w1 += static_cast<long long>(wh) * wl;
        w0 += static_cast<long long>(wl) * wl;
      }
      const __int128 sg = (static_cast<__int128>(g2) << 56) + (static_cast<__int128>(g1) << 28) + g0;
      const __int128 sw = (static_cast<__int128>(w2) << 58) + (static_cast<__int128>(w1) << 30) + w0;
      block_reduce_int(s0, s1, sg, sw, G, half_gamma_over_h2, out2);
    } else {
      double m = 0.0, ew = 0.0, eg = 0.0;
      for (int idx = threadIdx.x; idx < kTY * kTX; idx += kThreads) {
        const int r = idx / kTX, c = idx - r * kTX;
        const int hidx = (r + 2) * HC + (c + 2);
        const double u = sc[hidx];
        double lap;
        if (dig) {
          int q0, q1;
          lap5_digits(sb, hidx, HC, q0, q1);
          lap = ixd::ixi_combine<28>(q0, q1, w4);
        } else {
          lap = lap5(sc, hidx, HC);
        }
        const double w = fma(u, u, -1.0);
        m += u;
        ew = fma(w, w, ew);
        eg = fma(u, lap, eg);
      }
      block_reduce2<T>(m, fma(0.25, ew, -half_gamma_over_h2 * eg), out2);
    }
  }
}

// Fixed-order sum of the per-block partials -> out2 = (h^2 sum C, h^2 sum energy density).
__global__ void k_reduce_final(const double* __restrict__ partials, int nblocks, double h2,
                               double* __restrict__ out2) {
  __shared__ double sm[256], se[256];
  double m = 0.0, e = 0.0;
  for (int b = threadIdx.x; b < nblocks; b += 256) {
    m += partials[2 * b];
    e += partials[2 * b + 1];
  }
  sm[threadIdx.x] = m;
  se[threadIdx.x] = e;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      sm[threadIdx.x] += sm[threadIdx.x + s];
      se[threadIdx.x] += se[threadIdx.x + s];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out2[0] = h2 * sm[0];
    out2[1] = h2 * se[0];
  }
}

// ---- line solves (cs_penta.cuh) ---------------------------------------------------------------------
// A line's tables on the device: the table rows and the bias terms of phase 2, and the 8 P
// matrices of the chunk scan.
struct LineTab {
  const pn::TabRow* tab;
  const uint64_t* base;
  const double* mats;
};

// Accessors of one thread's chunk: 8 consecutive 64-bit words.
struct AccRow {  // words in a row, 16-byte aligned (shared memory)
  uint64_t* p;
  __device__ __forceinline__ void load8(int k, uint64_t (&v)[8]) const {
#pragma unroll
    for (int u = 0; u < 8; u += 2) {
      const ulonglong2 d = *reinterpret_cast<const ulonglong2*>(p + k + u);
      v[u] = d.x;
      v[u + 1] = d.y;
    }
  }
  __device__ __forceinline__ void store8(int k, const uint64_t (&v)[8]) const {
#pragma unroll
    for (int u = 0; u < 8; u += 2) *reinterpret_cast<ulonglong2*>(p + k + u) = make_ulonglong2(v[u], v[u + 1]);
  }
  __device__ __forceinline__ uint64_t get(int k) const { return p[k]; }
  __device__ __forceinline__ void put(int k, uint64_t v) const { p[k] = v; }
};
struct AccStride {  // words es apart (shared or global memory)
  uint64_t* p;
  int64_t es;
  __device__ __forceinline__ void load8(int k, uint64_t (&v)[8]) const {
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = p[(k + u) * es];
  }
  __device__ __forceinline__ void store8(int k, const uint64_t (&v)[8]) const {
#pragma unroll
    for (int u = 0; u < 8; ++u) p[(k + u) * es] = v[u];
  }
  __device__ __forceinline__ uint64_t get(int k) const { return p[k * es]; }
  __device__ __forceinline__ void put(int k, uint64_t v) const { p[k * es] = v; }
};
// 32-byte global accesses: a whole sector per thread and instruction
__device__ __forceinline__ void ld_words4(const uint64_t* p, uint64_t& a, uint64_t& b, uint64_t& c, uint64_t& d) {
  asm volatile("ld.global.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(a), "=l"(b), "=l"(c), "=l"(d) : "l"(p) : "memory");
}
__device__ __forceinline__ void st_words4(uint64_t* p, uint64_t a, uint64_t b, uint64_t c, uint64_t d) {
  asm volatile("st.global.v4.u64 [%0], {%1, %2, %3, %4};" ::"l"(p), "l"(a), "l"(b), "l"(c), "l"(d) : "memory");
}
struct AccWide {  // words in a row of global memory, 32-byte aligned
  uint64_t* p;
  int64_t es;
  __device__ __forceinline__ void load8(int k, uint64_t (&v)[8]) const {
    ld_words4(p + k, v[0], v[1], v[2], v[3]);
    ld_words4(p + k + 4, v[4], v[5], v[6], v[7]);
  }
  __device__ __forceinline__ void store8(int k, const uint64_t (&v)[8]) const {
    st_words4(p + k, v[0], v[1], v[2], v[3]);
    st_words4(p + k + 4, v[4], v[5], v[6], v[7]);
  }
  __device__ __forceinline__ uint64_t get(int k) const { return p[k]; }
  __device__ __forceinline__ void put(int k, uint64_t v) const { p[k] = v; }
};
template <int ES>
struct AccCols {  // ES columns interleaved (shared memory)
  uint64_t* p;
  __device__ __forceinline__ void load8(int k, uint64_t (&v)[8]) const {
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = p[(k + u) * ES];
  }
  __device__ __forceinline__ void store8(int k, const uint64_t (&v)[8]) const {
#pragma unroll
    for (int u = 0; u < 8; ++u) p[(k + u) * ES] = v[u];
  }
  __device__ __forceinline__ uint64_t get(int k) const { return p[k * ES]; }
  __device__ __forceinline__ void put(int k, uint64_t v) const { p[k * ES] = v; }
};

// The states entering chunk p of a line from all its chunks' end values: inclusive scans over the
// chunks with the recursion's own matrices, forward states then backward ones.  Every thread of the
// block calls it, P threads per line; sh: P double2 of the line.  The order of operations is
// reduce_host's.
template <bool NF>
__device__ __forceinline__ void reduce_states(const pn::Par& q, const double* __restrict__ mats, int P, int p,
                                              double2* sh, const double (&ends)[4], double (&st)[4]) {
  const bool cyclic = !NF && q.cyclic;
  auto scan = [&](bool fwd, double& a, double& b) {
#pragma unroll 1
    for (int l = 0; (1 << l) < P && l < q.levels; ++l) {
      int o = fwd ? p - (1 << l) : p + (1 << l);
      if (cyclic) o = o < 0 ? o + P : (o >= P ? o - P : o);
      sh[p] = make_double2(a, b);
      __syncthreads();
      if (o >= 0 && o < P) {
        const double2 v = sh[o];
        pn::mv_add(q.Ml[l], v.x, v.y, a, b, a, b);
      }
      __syncthreads();
    }
    sh[p] = make_double2(a, b);
    __syncthreads();
  };
  // a value that is not finite reaches every chunk of its line, as it would with every level
  auto finite = [](double x) { return ((pn::hi32(pn::dbits(x)) >> 20) & 0x7ffu) != 0x7ffu; };
  const bool own = finite(ends[0]) && finite(ends[1]) && finite(ends[2]) && finite(ends[3]);
  const bool broken = __syncthreads_or(!own);  // uniform over the block
  bool line_broken = false;
  if (broken) {
    sh[p] = make_double2(own ? 0.0 : 1.0, 0.0);
    __syncthreads();
    for (int k = 0; k < P; ++k) line_broken = line_broken || sh[k].x != 0.0;
    __syncthreads();
  }
  double a = ends[0], b = ends[1];
  scan(true, a, b);
  const double2 last = sh[P - 1];
  const int o = p > 0 ? p - 1 : P - 1;
  const double2 before = sh[o];
  double y0 = 0.0, y1 = 0.0;
  if (cyclic) {
    y0 = before.x;
    y1 = before.y;
  } else if constexpr (!NF) {
    double t0, t1;
    pn::mv_add(q.C, last.x, last.y, 0.0, 0.0, t0, t1);
    pn::mv_add(mats + 8 * o, t0, t1, before.x, before.y, y0, y1);
  } else if (p > 0) {
    y0 = before.x;
    y1 = before.y;
  }
  __syncthreads();
  pn::mv_add(q.R, y0, y1, ends[2], ends[3], a, b);
  if constexpr (NF) {
    if (p == P - 1) {
      double w0, w1;
      pn::mv_add(q.V, last.x, last.y, 0.0, 0.0, w0, w1);
      pn::mv_add(q.M, w0, w1, a, b, a, b);
    }
  }
  scan(false, a, b);
  const double2 first = sh[0];
  const int nx = p + 1 < P ? p + 1 : 0;
  const double2 after = sh[nx];
  double z0, z1;
  if (cyclic) {
    st[2] = after.x;
    st[3] = after.y;
  } else if constexpr (!NF) {
    pn::mv_add(q.C, first.x, first.y, 0.0, 0.0, z0, z1);
    pn::mv_add(mats + 8 * (P - 1 - nx), z0, z1, after.x, after.y, st[2], st[3]);
  } else {
    pn::mv_add(q.Z, first.x, first.y, 0.0, 0.0, z0, z1);
    if (p > 0) pn::mv_add(mats + 8 * (p - 1), z0, z1, y0, y1, y0, y1);
    else { y0 = z0; y1 = z1; }
    if (p + 1 < P) {
      pn::mv_add(mats + 8 * nx + 4, z0, z1, after.x, after.y, st[2], st[3]);
    } else {
      double t0, t1;
      pn::mv_add(mats + 8 * (P - 1), z0, z1, last.x, last.y, t0, t1);
      pn::mv_add(q.V, t0, t1, 0.0, 0.0, st[2], st[3]);
    }
  }
  st[0] = y0;
  st[1] = y1;
  if (line_broken) st[0] = st[1] = st[2] = st[3] = pn::from_bits(0x7ff8000000000000ull);
}

__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory"); }

// The table rows of phase 2, the same for every thread: from shared memory in the kernels that stage
// them (from global memory their latency bounded phase 2: 108 cycles a point and warp scheduler,
// 62 from shared memory), through the read-only cache otherwise.
struct TabShared {
  const ulonglong2* t;
  const uint64_t* b;
  __device__ __forceinline__ void row(int k, uint64_t (&v)[4], uint64_t& base) const {
    const ulonglong2 x = t[2 * k], y = t[2 * k + 1];
    v[0] = x.x; v[1] = x.y; v[2] = y.x; v[3] = y.y;
    base = b[k];
  }
};
struct TabGlobal {
  const ulonglong2* t;
  const unsigned long long* b;
  __device__ __forceinline__ explicit TabGlobal(const LineTab& lt)
      : t(reinterpret_cast<const ulonglong2*>(lt.tab)), b(reinterpret_cast<const unsigned long long*>(lt.base)) {}
  __device__ __forceinline__ void row(int k, uint64_t (&v)[4], uint64_t& base) const {
    const ulonglong2 x = __ldg(t + 2 * k), y = __ldg(t + 2 * k + 1);
    v[0] = x.x; v[1] = x.y; v[2] = y.x; v[3] = y.y;
    base = __ldg(b + k);
  }
};
constexpr int kTabBytes = 40;  // per point of a chunk

// Starts the copy of the tables to shared memory (16-byte aligned, kTabBytes m): rows, then bias
// terms.  The caller waits for it with its other copies.
__device__ __forceinline__ TabShared stage_tables(uint64_t* to, const LineTab& lt, int m) {
  for (int i = threadIdx.x; i < 2 * m; i += blockDim.x) cp_async16(to + 2 * i, reinterpret_cast<const uint64_t*>(lt.tab) + 2 * i);
  for (int i = threadIdx.x; i < m; i += blockDim.x) cp_async8(to + 4 * m + i, lt.base + i);
  return {reinterpret_cast<const ulonglong2*>(to), to + 4 * m};
}

// Phase 2 on a thread's chunk: every word of s (W at scale mark ew) becomes x, as a double's bits.
template <class Tab, class Acc>
__device__ __forceinline__ void correct_chunk(const pn::Par& q, const Tab& tab, const Acc& s, int m, int ew,
                                              const double (&st)[4]) {
  pn::Corr c;
  if (pn::corr_setup(q, ew, st, c)) {
    auto point = [&](int k, uint64_t w) {
      uint64_t t[4], b;
      tab.row(k, t, b);
      return pn::dbits(pn::from_fixed(pn::corr_point(c, w, t, b), c.eo));
    };
    for (int k0 = 0; k0 + 8 <= m; k0 += 8) {
      uint64_t v[8];
      s.load8(k0, v);
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = point(k0 + u, v[u]);
      s.store8(k0, v);
    }
    for (int k = m & ~7; k < m; ++k) s.put(k, point(k, s.get(k)));
    return;
  }
  if (st[0] != st[0]) {  // a line with a non-finite value (reduce_states): every point
#pragma unroll 1
    for (int k = 0; k < m; ++k) s.put(k, 0x7ff8000000000000ull);
    return;
  }
#pragma unroll 1
  for (int k = 0; k < m; ++k) {
    uint64_t t[4], b;
    tab.row(k, t, b);
    s.put(k, pn::dbits(pn::corr_native(q, ew, s.get(k), t, st)));
  }
}

// C^{n+1} = Cbar + v of one point: next holds Cbar = 2 C^n - C^{n-1}, written there by this step's
// right-hand side kernel (FP32 storage: formed in FP32, one rounding of the size of the result's own).
__device__ __forceinline__ double updated(double cbar, double v) { return cbar + v; }
__device__ __forceinline__ float updated(float cbar, double v) { return narrow_rn(widen(cbar) + v); }

// Words from one chunk to the next in shared memory: rows 2 modulo 4 (the lanes' 16-byte accesses then
// fall on different banks), columns an odd number of rows.
__host__ __device__ __forceinline__ int row_pitch(int m) { return m + ((6 - (m & 3)) & 3); }
__host__ __device__ __forceinline__ int col_pitch(int m) { return m | 1; }

// Whole lines in shared memory, both phases in one launch: the field is read once and written once.
// Rows: a few rows of n = P m values per block, one thread per (row, chunk).
template <bool NF>
__global__ void __launch_bounds__(64)
    k_line_rows(const double* __restrict__ in, double* __restrict__ out, const pn::Par q,
                            const LineTab lt, int P, int m, int vec) {
  extern __shared__ __align__(16) uint64_t sm[];
  const int chunks = blockDim.x, pitch = row_pitch(m);  // rows * P
  double2* sh = reinterpret_cast<double2*>(sm + static_cast<size_t>(chunks) * pitch);
  const TabShared tab = stage_tables(reinterpret_cast<uint64_t*>(sh + chunks), lt, m);
  const int64_t base = static_cast<int64_t>(blockIdx.x) * chunks * m;  // consecutive rows are one range
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
  const int lanes = min(32, static_cast<int>(blockDim.x) - 32 * warp);
  for (int c = warp; c < chunks; c += nw) {
    uint64_t* d = sm + c * pitch;
    const double* g = in + base + static_cast<int64_t>(c) * m;
    if (vec)
      for (int k = 2 * lane; k < m; k += 2 * lanes) cp_async16(d + k, g + k);
    else
      for (int k = lane; k < m; k += lanes) cp_async8(d + k, g + k);
  }
  cp_async_wait();
  __syncthreads();
  const int p = threadIdx.x % P;
  AccRow s{sm + threadIdx.x * pitch};
  double ends[4], st[4];
  const int ew = pn::local_solve(q, s, s, m, ends);
  reduce_states<NF>(q, lt.mats, P, p, sh + (threadIdx.x - p), ends, st);
  correct_chunk(q, tab, s, m, ew, st);
  __syncthreads();
  for (int c = warp; c < chunks; c += nw) {
    const double* d = reinterpret_cast<const double*>(sm + c * pitch);
    double* g = out + base + static_cast<int64_t>(c) * m;
    if (vec)
      for (int k = 2 * lane; k < m; k += 2 * lanes) *reinterpret_cast<double2*>(g + k) = *reinterpret_cast<const double2*>(d + k);
    else
      for (int k = lane; k < m; k += lanes) g[k] = d[k];
  }
}

// Columns: a cluster of CS blocks holds NC neighbouring columns, each block the n / CS rows of its
// chunks, so that every row is an 8 NC-byte piece (whole 128-byte lines for NC = 16: with two columns
// per block the 16-byte pieces alone took 0.35 ms at 4096^2) and a block still fits three to an
// SM.  Threads are (chunk, column), columns fastest.  Each block forms the entering states of NC / CS of
// the columns from all chunks' end values, read from and returned to the other blocks' shared
// memory.  The update C^{n+1} = Cbar + v is fused into the write.
template <int NC, typename T, bool NF>
__global__ void __launch_bounds__(256)
    k_line_cols(const double* __restrict__ in, T* __restrict__ next, int64_t n, const pn::Par q,
                const LineTab lt, int P, int m, int vec) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) uint64_t sm[];
  constexpr int H = NC / 2;
  cg::cluster_group cluster = cg::this_cluster();
  const int CS = static_cast<int>(cluster.num_blocks()), rank = static_cast<int>(cluster.block_rank());
  const int Pc = P / CS, threads = static_cast<int>(blockDim.x), pitch = col_pitch(m) * NC;  // Pc * NC threads
  // after the data: the scan's double2 per thread, then the end values (later the states), 4 per thread
  double2* sh = reinterpret_cast<double2*>(sm + static_cast<size_t>(Pc) * pitch);
  double* ex = reinterpret_cast<double*>(sh + threads);
  const TabShared tab = stage_tables(reinterpret_cast<uint64_t*>(ex + 4 * threads), lt, m);
  const int64_t x0 = static_cast<int64_t>(blockIdx.x / CS) * NC;
  const int64_t row0 = static_cast<int64_t>(rank) * Pc * m;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (threads + 31) >> 5;
  const int lanes = min(32, threads - 32 * warp);
  for (int c = warp; c < Pc; c += nw) {
    uint64_t* d = sm + c * pitch;
    const double* g = in + (row0 + static_cast<int64_t>(c) * m) * n + x0;
    for (int i = lane; i < m * H; i += lanes) cp_async16(d + 2 * i, g + static_cast<int64_t>(i / H) * n + 2 * (i % H));
  }
  cp_async_wait();
  __syncthreads();
  const int l = threadIdx.x % NC, c = threadIdx.x / NC;
  AccCols<NC> s{sm + c * pitch + l};
  double ends[4], st[4];
  const int ew = pn::local_solve(q, s, s, m, ends);
#pragma unroll
  for (int j = 0; j < 4; ++j) ex[j * threads + threadIdx.x] = ends[j];
  cluster.sync();
  {
    // this block's share of the columns, P threads each: chunk p of column rl is thread
    // (p % Pc) NC + rl of block p / Pc
    const int rl = rank * (NC / CS) + threadIdx.x / P, p = threadIdx.x % P;
    double* far = cluster.map_shared_rank(ex, p / Pc) + (p % Pc) * NC + rl;
#pragma unroll
    for (int j = 0; j < 4; ++j) ends[j] = far[j * threads];
    reduce_states<NF>(q, lt.mats, P, p, sh + (threadIdx.x - p), ends, st);
#pragma unroll
    for (int j = 0; j < 4; ++j) far[j * threads] = st[j];
  }
  cluster.sync();
#pragma unroll
  for (int j = 0; j < 4; ++j) st[j] = ex[j * threads + threadIdx.x];
  correct_chunk(q, tab, s, m, ew, st);
  __syncthreads();
  for (int cc = warp; cc < Pc; cc += nw) {
    const double* d = reinterpret_cast<const double*>(sm + cc * pitch);
    T* g = next + (row0 + static_cast<int64_t>(cc) * m) * n + x0;
    for (int i0 = lane; i0 < m * H; i0 += 4 * lanes) {  // four pieces in flight
      using V = typename std::conditional<sizeof(T) == 8, double2, float2>::type;
      V cb[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int i = i0 + j * lanes;
        if (i < m * H) {
          const T* a = g + static_cast<int64_t>(i / H) * n + 2 * (i % H);
          if (vec) cb[j] = *reinterpret_cast<const V*>(a);
          else { cb[j].x = a[0]; cb[j].y = a[1]; }
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int i = i0 + j * lanes;
        if (i < m * H) {
          T* a = g + static_cast<int64_t>(i / H) * n + 2 * (i % H);
          V r;
          r.x = updated(cb[j].x, d[2 * i]);
          r.y = updated(cb[j].y, d[2 * i + 1]);
          if (vec) *reinterpret_cast<V*>(a) = r;
          else { a[0] = r.x; a[1] = r.y; }
        }
      }
    }
  }
}

// Lines too long for shared memory, and the columns of a row band (whose chunks lie on several ranks):
// the two phases as kernels over global memory, one thread per (line, chunk), with the same
// functions, so the same values.  G holds W, scale the chunks' scale marks.
// Acc: AccWide for rows whose chunks are 32-byte aligned, else AccStride.
template <class Acc>
__global__ void __launch_bounds__(kSolveThreads)
    k_line_local(const double* __restrict__ in, uint64_t* __restrict__ G, double* __restrict__ bnd,
                 int* __restrict__ scale, const pn::Par q, int64_t lines, int Pl, int m, int64_t line_stride,
                 int64_t elem_stride) {
  const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= lines * Pl) return;
  const int64_t line = t % lines, pl = t / lines;
  const int64_t at = line * line_stride + pl * m * elem_stride;
  const Acc si{const_cast<uint64_t*>(reinterpret_cast<const uint64_t*>(in)) + at, elem_stride};
  const Acc s{G + at, elem_stride};
  double ends[4];
  scale[pl * lines + line] = pn::local_solve(q, si, s, m, ends);
#pragma unroll
  for (int j = 0; j < 4; ++j) bnd[(4 * pl + j) * lines + line] = ends[j];
}

// The states entering every chunk of every line: blocks of 8 lines x P chunks.
template <bool NF>
__global__ void __launch_bounds__(8 * pn::kMaxChunks)
    k_line_states(const double* __restrict__ bnd, double* __restrict__ states, const pn::Par q,
                              const LineTab lt, int64_t lines, int P) {
  extern __shared__ __align__(16) uint64_t sm[];
  const int l = threadIdx.x % 8, p = threadIdx.x / 8;
  const int64_t line = static_cast<int64_t>(blockIdx.x) * 8 + l;
  double ends[4] = {0.0, 0.0, 0.0, 0.0}, st[4];
  if (line < lines)
    for (int j = 0; j < 4; ++j) ends[j] = bnd[(4 * static_cast<int64_t>(p) + j) * lines + line];
  reduce_states<NF>(q, lt.mats, P, p, reinterpret_cast<double2*>(sm) + l * P, ends, st);
  if (line < lines)
    for (int j = 0; j < 4; ++j) states[(4 * static_cast<int64_t>(p) + j) * lines + line] = st[j];
}

template <int MODE, typename T, bool WIDE>
struct AccOut {  // reads W, writes the result of phase 2
  const uint64_t* p;
  double* out;
  T* next;
  int64_t es;
  __device__ __forceinline__ void load8(int k, uint64_t (&v)[8]) const {
    if constexpr (WIDE) {
      AccWide{const_cast<uint64_t*>(p), 1}.load8(k, v);
    } else {
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = p[(k + u) * es];
    }
  }
  __device__ __forceinline__ void store8(int k, const uint64_t (&v)[8]) const {
    if constexpr (MODE == 0 && WIDE) {
      AccWide{reinterpret_cast<uint64_t*>(out), 1}.store8(k, v);
    } else if constexpr (MODE == 0) {
#pragma unroll
      for (int u = 0; u < 8; ++u) out[(k + u) * es] = pn::from_bits(v[u]);
    } else {
      T cb[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) cb[u] = next[(k + u) * es];
#pragma unroll
      for (int u = 0; u < 8; ++u) next[(k + u) * es] = updated(cb[u], pn::from_bits(v[u]));
    }
  }
  __device__ __forceinline__ uint64_t get(int k) const { return p[k * es]; }
  __device__ __forceinline__ void put(int k, uint64_t v) const {
    if constexpr (MODE == 0) out[k * es] = pn::from_bits(v);
    else next[k * es] = updated(next[k * es], pn::from_bits(v));
  }
};

// MODE 0 writes x (FP64) to out; MODE 1 adds it to Cbar in next.
template <int MODE, typename T, bool WIDE = false>
__global__ void __launch_bounds__(kSolveThreads)
    k_line_correct(uint64_t* __restrict__ G, const double* __restrict__ states, const int* __restrict__ scale,
                   const pn::Par q, const LineTab lt, int64_t lines, int p0, int Pl, int m, int64_t line_stride,
                   int64_t elem_stride, double* __restrict__ out, T* __restrict__ next) {
  const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= lines * Pl) return;
  const int64_t line = t % lines, pl = t / lines;
  const int64_t at = line * line_stride + pl * m * elem_stride;
  AccOut<MODE, T, WIDE> s{G + at, MODE == 0 ? out + at : nullptr, MODE == 1 ? next + at : nullptr, elem_stride};
  double st[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) st[j] = states[(4 * (p0 + pl) + j) * lines + line];
  correct_chunk(q, TabGlobal(lt), s, m, scale[pl * lines + line], st);
}

// Valid partition: P divides n, chunks of at least 16 points, in whole register batches or (the solves
// take the last m % 8 points one by one) any power of two of them on the grids of 64 points' multiples.
bool whole_batches(int64_t n, int P) { return P >= 1 && n % P == 0 && (n / P) % kU == 0; }
bool valid_chunks(int64_t n, int P) {
  return P >= 1 && P <= pn::kMaxChunks && n % P == 0 && n / P >= 16 &&
         (whole_batches(n, P) || (n % 64 == 0 && (P & (P - 1)) == 0));
}

// Chunks of at least 16 points up to 32 chunks a line, of at least 32 beyond: the threads of a line
// are its chunks, and the scan over them costs what a few points do.  Rows + columns on GB300: 512^2
// 34 us with 32 chunks (39 with 16), 1024^2 48 us with 32 (54 with 16, 56 with 64), 2048^2 114 us with
// 64 (130 with 32), 4096^2 384 us with 64 (526 with 32).
// Where that leaves chunks of more than 64 points (n = 64 times an odd number), any chunk length.
int default_chunks(int64_t n) {
  auto longest = [&](bool any) {
    int P = 1;
    while (2 * P <= pn::kMaxChunks && n % (2 * P) == 0 && (any || whole_batches(n, 2 * P)) &&
           n / (2 * P) >= (P < 32 ? 16 : 32))
      P *= 2;
    return P;
  };
  const int P = longest(false);
  return n / P <= 64 ? P : longest(true);
}

// Tuning key of the partition.  Not the former solver's "ch|...": its best chunk counts (16 at 4096^2), saved in a
// file, would keep this one from its own.
std::string partition_key(int storage, bool noflux, int64_t n) {
  char key[96];
  snprintf(key, sizeof key, "chlines|%s%s|n%lld|sm%d", storage == CS_F32 ? "f32" : "f64", noflux ? "|noflux" : "",
           (long long)n, num_sms());
  return key;
}

// FP64 tiles (C^n, Cbar: halo 2; Z: halo 1), for either storage type.
size_t rhs_smem_bytes() {
  return 8 * (2 * (kTY + 4) * (kTX + 4));  // C^n and Cbar (Z reuses Cbar's space)
}

template <typename T> int set_rhs_attr() {
  static bool done = false;
  if (!done) {
    const int bytes = static_cast<int>(rhs_smem_bytes());
    CS_CUDA_TRY(cudaFuncSetAttribute(k_ch_rhs<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    done = true;
  }
  return CS_OK;
}

template <typename T>
int launch_rhs(CHPlan* p, bool with_rhs, double* partials, cudaStream_t s) {
  int rc = set_rhs_attr<T>();
  if (rc != CS_OK) return rc;
  dim3 grid(static_cast<unsigned>(p->n / kTX), static_cast<unsigned>(p->n / kTY));
  const T* cur = static_cast<const T*>(p->field[p->icur]);
  const T* prev = static_cast<const T*>(p->field[p->iprev]);
  double* rhs = with_rhs ? p->A : nullptr;
  T* cbar = with_rhs ? static_cast<T*>(p->field[p->inext]) : nullptr;
  k_ch_rhs<T><<<grid, kThreads, rhs_smem_bytes(), s>>>(cur, prev, rhs, p->n, p->alpha, p->a,
                                                        0.5 * p->gamma / (p->h * p->h), partials, p->noflux,
                                                        ixd::ixi_round51(-p->a),
                                                        cubic_inv(p->alpha, ixd::ixi_round51(-p->a)), 0, cbar);
  CS_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  return CS_OK;
}

LineTab line_tab(const Lines& L) {
  const pn::TabRow* tab = reinterpret_cast<const pn::TabRow*>(L.tables + static_cast<size_t>(8) * L.P);
  return {tab, reinterpret_cast<const uint64_t*>(tab + L.m), L.tables};
}
// scratch of the global-memory kernels for `lines` lines: end values, states, scale marks
size_t scratch_doubles(int64_t lines, int P) { return static_cast<size_t>(8) * P * lines + (static_cast<size_t>(P) * lines + 1) / 2; }
double* line_ends(const Lines& L) { return L.scratch; }
double* line_states(const Lines& L, int64_t lines) { return L.scratch + static_cast<size_t>(4) * L.P * lines; }
int* line_scale(const Lines& L, int64_t lines) { return reinterpret_cast<int*>(L.scratch + static_cast<size_t>(8) * L.P * lines); }

void free_lines(Lines* L) {
  cudaFree(L->tables);
  cudaFree(L->scratch);
  L->tables = L->scratch = nullptr;
}

// Builds the solver for lines of n points in P chunks; scratch_lines > 0 also allocates the scratch.
int make_lines(int64_t n, int P, double a, bool noflux, int64_t scratch_lines, Lines* L) {
  std::vector<pn::TabRow> tab;
  std::vector<uint64_t> base;
  std::vector<double> mats;
  L->tables = L->scratch = nullptr;
  L->P = P;
  L->m = static_cast<int>(n / P);
  if (!pn::build(n, P, a, noflux, L->par, tab, base, mats))
    return set_error(CS_EINVAL, "Cahn-Hilliard line coefficient a = %g is outside the solver's range", a);
  const size_t nm = mats.size(), nt = 4 * tab.size(), nb = base.size();
  std::vector<double> all(nm + nt + nb);
  memcpy(all.data(), mats.data(), nm * 8);
  memcpy(all.data() + nm, tab.data(), nt * 8);
  memcpy(all.data() + nm + nt, base.data(), nb * 8);
  cudaError_t e = cudaMalloc(&L->tables, all.size() * 8);
  if (e == cudaSuccess && scratch_lines > 0) e = cudaMalloc(&L->scratch, scratch_doubles(scratch_lines, P) * 8);
  if (e == cudaSuccess) e = cudaMemcpy(L->tables, all.data(), all.size() * 8, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) return CS_OK;
  free_lines(L);
  return e == cudaErrorMemoryAllocation ? set_error(CS_ENOMEM, "Cahn-Hilliard line tables: %s", cudaGetErrorString(e))
                                        : cuda_error(e, "Cahn-Hilliard line tables");
}

// Shapes of the shared-memory kernels.  Blocks take at most kLineSmem bytes where they can, so that
// three or more share an SM and one's loads and stores run under the others' arithmetic.
constexpr size_t kLineSmem = 75 * 1024, kLineSmemMax = 220 * 1024;

// Rows per block (a row takes P row_pitch(m) words and the scan 2 P), 0 when a row does not fit; one or two
// warps per block.
size_t rows_smem(int P, int m, int k) { return static_cast<size_t>(k) * P * (8 * row_pitch(m) + 16) + kTabBytes * m; }
int rows_per_block(int64_t rows, int P, int m) {
  int k = 1;
  while (k * P < 32 && k < 32) k *= 2;
  while (k > 1 && (rows % k != 0 || rows_smem(P, m, k) > kLineSmem)) k /= 2;
  return rows_smem(P, m, k) <= kLineSmemMax ? k : 0;
}

// Columns per cluster and blocks per cluster, {0, 0} when they do not fit: as many blocks as divide
// the chunks (eight at most), sixteen columns when that fits kLineSmem, else eight.
struct ColShape { int nc, cs; };
size_t cols_smem(int P, int m, ColShape s) {
  return static_cast<size_t>(P / s.cs) * s.nc * (8 * col_pitch(m) + 16 + 32) + kTabBytes * m;
}
ColShape cols_shape(int P, int m) {
  int cs = 8;
  while (P % cs != 0) cs /= 2;
  const ColShape a{16, cs}, b{8, cs};
  auto fits = [&](ColShape s, size_t most) { return cols_smem(P, m, s) <= most && s.nc * (P / s.cs) <= 256; };
  if (fits(a, kLineSmem)) return a;
  if (fits(b, kLineSmemMax)) return b;
  return {0, 0};
}

// The states of `lines` lines from the end values of all their chunks, into the scratch.
void launch_states(const Lines& L, bool noflux, int64_t lines, const double* ends, cudaStream_t s) {
  const unsigned grid = static_cast<unsigned>((lines + 7) / 8);
  const size_t smem = static_cast<size_t>(8) * L.P * sizeof(double2);
  if (noflux) k_line_states<true><<<grid, 8 * L.P, smem, s>>>(ends, line_states(L, lines), L.par, line_tab(L), lines, L.P);
  else k_line_states<false><<<grid, 8 * L.P, smem, s>>>(ends, line_states(L, lines), L.par, line_tab(L), lines, L.P);
}

// Solves along the rows of `rows` x n values (out may equal in).  B: rows x n scratch, used only when a
// row does not fit in shared memory.
int launch_rows(const Lines& L, bool noflux, int64_t rows, const double* in, double* out, double* B, cudaStream_t s) {
  const int P = L.P, m = L.m;
  const int64_t n = static_cast<int64_t>(P) * m;
  const LineTab lt = line_tab(L);
  if (const int k = rows_per_block(rows, P, m)) {
    const int vec = ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15u) == 0 && m % 2 == 0;
    const unsigned grid = static_cast<unsigned>(rows / k);
    const size_t smem = rows_smem(P, m, k);
    if (noflux) k_line_rows<true><<<grid, k * P, smem, s>>>(in, out, L.par, lt, P, m, vec);
    else k_line_rows<false><<<grid, k * P, smem, s>>>(in, out, L.par, lt, P, m, vec);
    CS_CUDA_TRY(cudaGetLastError());
    count_launches(1);
    return CS_OK;
  }
  const unsigned grid = static_cast<unsigned>((rows * P + kSolveThreads - 1) / kSolveThreads);
  uint64_t* G = reinterpret_cast<uint64_t*>(B);
  // every chunk of a row (n is a multiple of 64) starts on a 32-byte boundary
  const bool wide = ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out) | reinterpret_cast<uintptr_t>(B)) & 31u) == 0 && m % 4 == 0;
  auto local = wide ? k_line_local<AccWide> : k_line_local<AccStride>;
  auto correct = wide ? k_line_correct<0, double, true> : k_line_correct<0, double, false>;
  local<<<grid, kSolveThreads, 0, s>>>(in, G, line_ends(L), line_scale(L, rows), L.par, rows, P, m, n, 1);
  launch_states(L, noflux, rows, line_ends(L), s);
  correct<<<grid, kSolveThreads, 0, s>>>(G, line_states(L, rows), line_scale(L, rows), L.par, lt, rows, 0, P, m, n, 1, out,
                                         static_cast<double*>(nullptr));
  CS_CUDA_TRY(cudaGetLastError());
  count_launches(3);
  return CS_OK;
}

// Solves along the columns of the n x n grid and adds the result to Cbar in next.
template <typename T>
int launch_cols(const Lines& L, bool noflux, const double* in, T* next, double* B, cudaStream_t s) {
  const int P = L.P, m = L.m;
  const int64_t n = static_cast<int64_t>(P) * m;
  const LineTab lt = line_tab(L);
  const ColShape sh = cols_shape(P, m);
  if (sh.nc) {
    const int vec = (reinterpret_cast<uintptr_t>(next) & (2 * sizeof(T) - 1)) == 0;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim = {static_cast<unsigned>(sh.cs), 1, 1};
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3(static_cast<unsigned>(n / sh.nc * sh.cs));
    cfg.blockDim = dim3(static_cast<unsigned>(sh.nc * (P / sh.cs)));
    cfg.dynamicSmemBytes = cols_smem(P, m, sh);
    cfg.stream = s;
    auto kern = noflux ? (sh.nc == 16 ? k_line_cols<16, T, true> : k_line_cols<8, T, true>)
                       : (sh.nc == 16 ? k_line_cols<16, T, false> : k_line_cols<8, T, false>);
    CS_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, in, next, n, L.par, lt, P, m, vec));
    count_launches(1);
    return CS_OK;
  }
  const unsigned grid = static_cast<unsigned>((n * P + kSolveThreads - 1) / kSolveThreads);
  k_line_local<AccStride><<<grid, kSolveThreads, 0, s>>>(in, reinterpret_cast<uint64_t*>(B), line_ends(L), line_scale(L, n), L.par, n, P,
                                              m, 1, n);
  launch_states(L, noflux, n, line_ends(L), s);
  k_line_correct<1, T><<<grid, kSolveThreads, 0, s>>>(reinterpret_cast<uint64_t*>(B), line_states(L, n), line_scale(L, n),
                                                      L.par, lt, n, 0, P, m, 1, n, nullptr, next);
  CS_CUDA_TRY(cudaGetLastError());
  count_launches(3);
  return CS_OK;
}

// The shared-memory kernels' size limit, set before any launch or capture.
int set_line_attrs() {
  const int bytes = static_cast<int>(kLineSmemMax);
  const void* kerns[] = {
      reinterpret_cast<const void*>(k_line_rows<false>), reinterpret_cast<const void*>(k_line_rows<true>),
#define CS_LINE_COLS(T, NF)                                   \
  reinterpret_cast<const void*>(k_line_cols<8, T, NF>), reinterpret_cast<const void*>(k_line_cols<16, T, NF>)
      CS_LINE_COLS(double, false), CS_LINE_COLS(double, true), CS_LINE_COLS(float, false), CS_LINE_COLS(float, true)
#undef CS_LINE_COLS
  };
  for (const void* k : kerns) CS_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  return CS_OK;
}

// Whether a full-grid plan needs the global-memory kernels' scratch.
bool needs_scratch(int64_t n, int P) {
  const int m = static_cast<int>(n / P);
  return !rows_per_block(n, P, m) || !cols_shape(P, m).nc;
}

template <typename T>
int launch_step(CHPlan* p, double* partials, cudaStream_t s) {
  int rc = launch_rhs<T>(p, true, partials, s);
  if (rc != CS_OK) return rc;
  rc = launch_rows(p->lines, p->noflux != 0, p->n, p->A, p->A, p->B, s);
  if (rc != CS_OK) return rc;
  return launch_cols<T>(p->lines, p->noflux != 0, p->A, static_cast<T*>(p->field[p->inext]), p->B, s);
}

void rotate(CHPlan* p) {
  const int old_prev = p->iprev;
  p->iprev = p->icur;
  p->icur = p->inext;
  p->inext = old_prev;
  ++p->steps;
}

int reduce_current(CHPlan* p, double* out2, cudaStream_t s) {
  int rc = p->storage == CS_F32 ? launch_rhs<float>(p, false, p->partials, s)
                                : launch_rhs<double>(p, false, p->partials, s);
  if (rc != CS_OK) return rc;
  k_reduce_final<<<1, 256, 0, s>>>(p->partials, p->rhs_blocks, p->h * p->h, out2);
  CS_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  return CS_OK;
}

void free_plan(CHPlan* p) {
  if (!p) return;
  drop_graphs(p);
  free_lines(&p->lines);
  cudaFree(p->A); cudaFree(p->B);
  cudaFree(p->partials); cudaFree(p->inv); cudaFree(p->diag);
  delete p;
}

}  // namespace

int ch_create(CHPlan** out, const cs_ch_desc* d, void* prev, void* cur, void* next) {
  *out = nullptr;
  if (!d) return set_error(CS_EINVAL, "null Cahn-Hilliard description");
  if (d->n < 64 || d->n % 64 != 0 || d->n > 65536)
    return set_error(CS_EINVAL, "n must be a multiple of 64 in [64, 65536]");
  if (d->storage != CS_F64 && d->storage != CS_F32) return set_error(CS_EINVAL, "storage must be CS_F64 or CS_F32");
  if (d->boundary != CS_CH_PERIODIC && d->boundary != CS_CH_NOFLUX)
    return set_error(CS_EINVAL, "boundary must be CS_CH_PERIODIC or CS_CH_NOFLUX");
  if (!(d->D > 0) || !(d->gamma >= 0) || !(d->dt > 0) || !std::isfinite(d->D) || !std::isfinite(d->gamma) || !std::isfinite(d->dt))
    return set_error(CS_EINVAL, "D > 0, gamma >= 0, dt > 0 and finite are required");
  if (!prev || !cur || !next) return set_error(CS_EINVAL, "null field buffer");
  const size_t eb = d->storage == CS_F32 ? 4 : 8;
  const size_t bytes = static_cast<size_t>(d->n) * d->n * eb;
  void* f[3] = {prev, cur, next};
  for (int i = 0; i < 3; ++i) {
    if (reinterpret_cast<uintptr_t>(f[i]) % eb) return set_error(CS_EINVAL, "fields must be aligned to the element size");
    for (int j = i + 1; j < 3; ++j) {
      const char* a = static_cast<const char*>(f[i]);
      const char* b = static_cast<const char*>(f[j]);
      if (a < b + bytes && b < a + bytes) return set_error(CS_EALIAS, "the three fields must not overlap");
    }
  }
  CHPlan* p = new (std::nothrow) CHPlan;
  if (!p) return set_error(CS_ENOMEM, "out of host memory");
  memset(p, 0, sizeof *p);
  p->n = d->n;
  p->storage = d->storage;
  p->noflux = d->boundary == CS_CH_NOFLUX;
  p->D = d->D; p->gamma = d->gamma; p->dt = d->dt;
  p->h = 2.0 * M_PI / static_cast<double>(d->n);
  const double h2 = p->h * p->h;
  p->a = (2.0 / 3.0) * d->D * d->gamma * d->dt / (h2 * h2);
  p->alpha = (2.0 / 3.0) * d->D * d->dt / h2;
  int P = default_chunks(d->n);
  int choice;
  if (tune_lookup(partition_key(d->storage, p->noflux, d->n), &choice) && valid_chunks(d->n, choice)) P = choice;
  p->P = P;
  p->m = static_cast<int>(d->n / P);
  p->field[0] = prev; p->field[1] = cur; p->field[2] = next;
  p->iprev = 0; p->icur = 1; p->inext = 2;
  p->rhs_blocks = static_cast<int>((d->n / kTX) * (d->n / kTY));
  int rc = make_lines(d->n, P, p->a, p->noflux != 0, needs_scratch(d->n, P) ? d->n : 0, &p->lines);
  if (rc != CS_OK) { free_plan(p); return rc; }
  const size_t nn = static_cast<size_t>(d->n) * d->n;
  cudaError_t e = cudaSuccess;
  if (e == cudaSuccess) e = cudaMalloc(&p->A, nn * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&p->B, nn * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&p->partials, static_cast<size_t>(2) * p->rhs_blocks * sizeof(double));
  if (e != cudaSuccess) {
    free_plan(p);
    return e == cudaErrorMemoryAllocation ? set_error(CS_ENOMEM, "Cahn-Hilliard workspace: %s", cudaGetErrorString(e))
                                          : cuda_error(e, "Cahn-Hilliard workspace");
  }
  rc = d->storage == CS_F32 ? set_rhs_attr<float>() : set_rhs_attr<double>();  // before any capture
  if (rc == CS_OK) rc = set_line_attrs();
  if (rc != CS_OK) { free_plan(p); return rc; }
  *out = p;
  return CS_OK;
}

void drop_graphs(CHPlan* p) {
  for (int i = 0; i < 3; ++i) {
    if (p->graph3[i]) cudaGraphExecDestroy(p->graph3[i]);
    p->graph3[i] = nullptr;
  }
}

// Captures three consecutive steps starting at the current rotation phase into a graph (the
// buffers return to the same roles after three steps, so the graph replays as is).
int capture_three(CHPlan* p, cudaGraphExec_t* out) {
  cudaStream_t cap;
  CS_CUDA_TRY(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
  const int ip = p->iprev, ic = p->icur, in = p->inext;
  const int64_t steps = p->steps;
  const int64_t before = cs_launch_count();
  cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
  int rc = e == cudaSuccess ? CS_OK : cuda_error(e, "cudaStreamBeginCapture");
  for (int k = 0; k < 3 && rc == CS_OK; ++k) {
    rc = p->storage == CS_F32 ? launch_step<float>(p, nullptr, cap) : launch_step<double>(p, nullptr, cap);
    rotate(p);
  }
  cudaGraph_t g = nullptr;
  cudaError_t e2 = cudaStreamEndCapture(cap, &g);
  cudaStreamDestroy(cap);
  p->iprev = ip; p->icur = ic; p->inext = in; p->steps = steps;  // capture ran nothing
  p->graph_kernels = static_cast<int>(cs_launch_count() - before);
  count_launches(-p->graph_kernels);
  if (rc != CS_OK) { if (g) cudaGraphDestroy(g); return rc; }
  if (e2 != cudaSuccess) return cuda_error(e2, "cudaStreamEndCapture");
  cudaError_t e3 = cudaGraphInstantiate(out, g, 0);
  cudaGraphDestroy(g);
  if (e3 != cudaSuccess) { *out = nullptr; return cuda_error(e3, "cudaGraphInstantiate"); }
  return CS_OK;
}

int ch_step(CHPlan* p, int64_t nsteps, double* h_mass, double* h_energy, cudaStream_t s) {
  if (nsteps < 0) return set_error(CS_EINVAL, "nsteps must be >= 0");
  if (nsteps == 0) return CS_OK;
  const bool want = h_mass || h_energy;
  if (!want) {  // blocks of three steps replay a captured graph (fewer launch gaps)
    while (nsteps >= 3) {
      cudaGraphExec_t& g = p->graph3[p->icur];
      if (!g) {
        int rc = capture_three(p, &g);
        if (rc != CS_OK) return rc;
      }
      CS_CUDA_TRY(cudaGraphLaunch(g, s));
      count_launches(p->graph_kernels);
      rotate(p); rotate(p); rotate(p);
      nsteps -= 3;
    }
    for (; nsteps > 0; --nsteps) {
      int rc = p->storage == CS_F32 ? launch_step<float>(p, nullptr, s) : launch_step<double>(p, nullptr, s);
      if (rc != CS_OK) return rc;
      rotate(p);
    }
    return CS_OK;
  }
  if (p->inv_cap < nsteps) {
    if (p->inv) cudaFree(p->inv);
    p->inv = nullptr;
    p->inv_cap = 0;
    cudaError_t e = cudaMalloc(&p->inv, static_cast<size_t>(2) * nsteps * sizeof(double));
    if (e != cudaSuccess) return cuda_error(e, "invariant buffer");
    p->inv_cap = nsteps;
  }
  for (int64_t st = 0; st < nsteps; ++st) {
    // the RHS kernel of step st reads C^n = the field after step st-1: reduce it on the way
    double* part = st > 0 ? p->partials : nullptr;
    int rc = p->storage == CS_F32 ? launch_step<float>(p, part, s) : launch_step<double>(p, part, s);
    if (rc != CS_OK) return rc;
    if (part) {
      // partials were consumed into a fixed-order sum before the next RHS overwrites them
      k_reduce_final<<<1, 256, 0, s>>>(p->partials, p->rhs_blocks, p->h * p->h, p->inv + 2 * (st - 1));
      CS_CUDA_TRY(cudaGetLastError());
      count_launches(1);
    }
    rotate(p);
  }
  int rc = reduce_current(p, p->inv + 2 * (nsteps - 1), s);
  if (rc != CS_OK) return rc;
  std::vector<double> h(static_cast<size_t>(2) * nsteps);
  CS_CUDA_TRY(cudaMemcpyAsync(h.data(), p->inv, h.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
  CS_CUDA_TRY(cudaStreamSynchronize(s));
  for (int64_t st = 0; st < nsteps; ++st) {
    if (h_mass) h_mass[st] = h[2 * st];
    if (h_energy) h_energy[st] = h[2 * st + 1];
  }
  return CS_OK;
}

int ch_invariants(CHPlan* p, double* mass, double* energy, cudaStream_t s) {
  if (p->inv_cap < 1) {
    cudaError_t e = cudaMalloc(&p->inv, 2 * sizeof(double));
    if (e != cudaSuccess) return cuda_error(e, "invariant buffer");
    p->inv_cap = 1;
  }
  int rc = reduce_current(p, p->inv, s);
  if (rc != CS_OK) return rc;
  double h[2];
  CS_CUDA_TRY(cudaMemcpyAsync(h, p->inv, sizeof h, cudaMemcpyDeviceToHost, s));
  CS_CUDA_TRY(cudaStreamSynchronize(s));
  if (mass) *mass = h[0];
  if (energy) *energy = h[1];
  return CS_OK;
}

namespace {

// ---- coarsening measures (Sec. 5.1, "Numerical Results") ---------------------------------------
//   s(t)   = 1 / (1 - <C^2>), <.> the spatial average by Simpson's rule on the periodic grid
//            (weights 2, 4, 2, 4, ... per direction: the end point 2 pi is the start point);
//   k_1(t) = sum_k |C^(k)|^2 / sum_k |k|^-1 |C^(k)|^2 over the discrete wavenumbers, k = 0 left out
//            (the k-space integrals with their common measure cancelled).
// The 2D DFT is two passes of a radix-2 FFT (one CTA per row, the row in shared memory): the
// first transforms the rows of C and writes them transposed into the (A, B) = (re, im) scratch,
// the second transforms those rows (the columns of C) and sums the spectrum.  All FP64.

constexpr int kDiagThreads = 256;

template <typename T>
__global__ void __launch_bounds__(kDiagThreads)
    k_simpson_rows(const T* __restrict__ c, int64_t n, double* __restrict__ partials) {
  const int64_t j = blockIdx.x;  // one row per block
  double acc = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += kDiagThreads) {
    const double v = widen(c[j * n + i]);
    acc += ((i & 1) ? 4.0 : 2.0) * v * v;
  }
  __shared__ double red[kDiagThreads / 32];
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double r = 0.0;
    for (int w = 0; w < kDiagThreads / 32; ++w) r += red[w];
    partials[j] = ((j & 1) ? 4.0 : 2.0) * r;
  }
}

// In-place radix-2 decimation-in-time FFT of the n = 2^logn points in (xr, xi) (shared memory,
// loaded in bit-reversed order); tw holds exp(-2 pi i t / n) for t < n / 2.
__device__ __forceinline__ void fft_smem(double* xr, double* xi, int n, int logn, const double2* __restrict__ tw) {
  for (int len = 2, stride = n >> 1; len <= n; len <<= 1, stride >>= 1) {
    const int half = len >> 1;
    for (int b = threadIdx.x; b < (n >> 1); b += kDiagThreads) {
      const int pos = b & (half - 1);
      const int i = (b - pos) * 2 + pos, k = i + half;
      const double2 w = tw[pos * stride];
      const double vr = w.x * xr[k] - w.y * xi[k];
      const double vi = w.x * xi[k] + w.y * xr[k];
      const double ur = xr[i], ui = xi[i];
      xr[i] = ur + vr;
      xi[i] = ui + vi;
      xr[k] = ur - vr;
      xi[k] = ui - vi;
    }
    __syncthreads();
  }
  (void)logn;
}

__device__ __forceinline__ int bit_reverse(int t, int logn) { return static_cast<int>(__brev(static_cast<unsigned>(t)) >> (32 - logn)); }

// Pass 1: the FFT of row j of C, written as column j of (re, im).
template <typename T>
__global__ void __launch_bounds__(kDiagThreads)
    k_fft_rows(const T* __restrict__ c, int n, int logn, const double2* __restrict__ tw,
               double* __restrict__ re, double* __restrict__ im) {
  extern __shared__ double xs[];
  double* xr = xs;
  double* xi = xs + n;
  const int64_t j = blockIdx.x;
  for (int t = threadIdx.x; t < n; t += kDiagThreads) {
    const int r = bit_reverse(t, logn);
    xr[r] = widen(c[j * n + t]);
    xi[r] = 0.0;
  }
  __syncthreads();
  fft_smem(xr, xi, n, logn, tw);
  for (int k = threadIdx.x; k < n; k += kDiagThreads) {
    re[static_cast<int64_t>(k) * n + j] = xr[k];
    im[static_cast<int64_t>(k) * n + j] = xi[k];
  }
}

// Pass 2: the FFT of row kx of (re, im) (column kx of the row transforms) gives C^(kx, ky) for
// every ky; the block sums |C^|^2 and |k|^-1 |C^|^2 (k = 0 left out) into partials[2 kx + 0/1].
__global__ void __launch_bounds__(kDiagThreads)
    k_fft_cols_spectrum(const double* __restrict__ re, const double* __restrict__ im, int n, int logn,
                        const double2* __restrict__ tw, double* __restrict__ partials) {
  extern __shared__ double xs[];
  double* xr = xs;
  double* xi = xs + n;
  const int kx = blockIdx.x;
  for (int t = threadIdx.x; t < n; t += kDiagThreads) {
    const int r = bit_reverse(t, logn);
    xr[r] = re[static_cast<int64_t>(kx) * n + t];
    xi[r] = im[static_cast<int64_t>(kx) * n + t];
  }
  __syncthreads();
  fft_smem(xr, xi, n, logn, tw);
  const double fx = kx <= n / 2 ? kx : kx - n;
  double num = 0.0, den = 0.0;
  for (int ky = threadIdx.x; ky < n; ky += kDiagThreads) {
    if (kx == 0 && ky == 0) continue;
    const double fy = ky <= n / 2 ? ky : ky - n;
    const double pw = xr[ky] * xr[ky] + xi[ky] * xi[ky];
    num += pw;
    den += pw / sqrt(fx * fx + fy * fy);
  }
  __shared__ double red[2][kDiagThreads / 32];
  for (int off = 16; off > 0; off >>= 1) {
    num += __shfl_down_sync(0xffffffffu, num, off);
    den += __shfl_down_sync(0xffffffffu, den, off);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = num;
    red[1][threadIdx.x >> 5] = den;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0;
    for (int w = 0; w < kDiagThreads / 32; ++w) {
      a += red[0][w];
      b += red[1][w];
    }
    partials[2 * kx] = a;
    partials[2 * kx + 1] = b;
  }
}

// Fixed-order sums of the partials: out[0] = sum of n Simpson row sums, out[1], out[2] = the two
// spectral sums.
__global__ void k_coarsening_final(const double* __restrict__ simpson, const double* __restrict__ spec,
                                   int n, double* __restrict__ out) {
  __shared__ double r[3][256];
  double a = 0.0, b = 0.0, c = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) {
    a += simpson[i];
    b += spec[2 * i];
    c += spec[2 * i + 1];
  }
  r[0][threadIdx.x] = a;
  r[1][threadIdx.x] = b;
  r[2][threadIdx.x] = c;
  __syncthreads();
  for (int st = 128; st > 0; st >>= 1) {
    if (threadIdx.x < st)
      for (int q = 0; q < 3; ++q) r[q][threadIdx.x] += r[q][threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int q = 0; q < 3; ++q) out[q] = r[q][0];
}

}  // namespace

int ch_coarsening(CHPlan* p, double* s_out, double* k1_out, cudaStream_t st) {
  if (p->noflux) return set_error(CS_EUNSUPPORTED, "the coarsening measures are defined on the periodic grid");
  const int64_t n = p->n;
  int logn = 0;
  while ((int64_t(1) << logn) < n) ++logn;
  if ((int64_t(1) << logn) != n) return set_error(CS_EUNSUPPORTED, "coarsening measures need n a power of two");
  const size_t smem = 2 * static_cast<size_t>(n) * sizeof(double);
  if (smem > 200 * 1024) return set_error(CS_EUNSUPPORTED, "n = %lld too large for the shared-memory FFT", (long long)n);
  // diag: [0, n) twiddles as n/2 (re, im) pairs, [n, 2n) Simpson row sums, [2n, 4n) spectrum sums, 4 results
  if (!p->diag) {
    std::vector<double> tw(static_cast<size_t>(n));
    for (int64_t t = 0; t < n / 2; ++t) {
      const double ang = -2.0 * M_PI * static_cast<double>(t) / static_cast<double>(n);
      tw[2 * t] = std::cos(ang);
      tw[2 * t + 1] = std::sin(ang);
    }
    double* d = nullptr;
    cudaError_t e = cudaMalloc(&d, (4 * static_cast<size_t>(n) + 4) * sizeof(double));
    if (e != cudaSuccess)
      return e == cudaErrorMemoryAllocation ? set_error(CS_ENOMEM, "coarsening buffers: %s", cudaGetErrorString(e))
                                            : cuda_error(e, "coarsening buffers");
    e = cudaMemcpyAsync(d, tw.data(), n * sizeof(double), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
      cudaFree(d);
      return cuda_error(e, "coarsening twiddles");
    }
    p->diag = d;
  }
  // the attribute is per function and process-wide: set it for this plan's n on every call
  CS_CUDA_TRY(cudaFuncSetAttribute(k_fft_rows<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)));
  CS_CUDA_TRY(cudaFuncSetAttribute(k_fft_rows<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)));
  CS_CUDA_TRY(cudaFuncSetAttribute(k_fft_cols_spectrum, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)));
  const double2* tw = reinterpret_cast<const double2*>(p->diag);
  double* simpson = p->diag + n;
  double* spec = p->diag + 2 * n;
  double* res = p->diag + 4 * n;
  const unsigned grid = static_cast<unsigned>(n);
  if (p->storage == CS_F32) {
    const float* c = static_cast<const float*>(p->field[p->icur]);
    k_simpson_rows<float><<<grid, kDiagThreads, 0, st>>>(c, n, simpson);
    k_fft_rows<float><<<grid, kDiagThreads, smem, st>>>(c, static_cast<int>(n), logn, tw, p->A, p->B);
  } else {
    const double* c = static_cast<const double*>(p->field[p->icur]);
    k_simpson_rows<double><<<grid, kDiagThreads, 0, st>>>(c, n, simpson);
    k_fft_rows<double><<<grid, kDiagThreads, smem, st>>>(c, static_cast<int>(n), logn, tw, p->A, p->B);
  }
  k_fft_cols_spectrum<<<grid, kDiagThreads, smem, st>>>(p->A, p->B, static_cast<int>(n), logn, tw, spec);
  k_coarsening_final<<<1, 256, 0, st>>>(simpson, spec, static_cast<int>(n), res);
  CS_CUDA_TRY(cudaGetLastError());
  count_launches(4);
  double h[3];
  CS_CUDA_TRY(cudaMemcpyAsync(h, res, sizeof h, cudaMemcpyDeviceToHost, st));
  CS_CUDA_TRY(cudaStreamSynchronize(st));
  const double mean_c2 = h[0] / (9.0 * static_cast<double>(n) * static_cast<double>(n));
  if (s_out) *s_out = 1.0 / (1.0 - mean_c2);
  if (k1_out) *k1_out = h[1] / h[2];
  return CS_OK;
}

int ch_fields(CHPlan* p, void** prev, void** cur, int64_t* steps) {
  if (prev) *prev = p->field[p->iprev];
  if (cur) *cur = p->field[p->icur];
  if (steps) *steps = p->steps;
  return CS_OK;
}

namespace {

// (Re)builds the line solver for P chunks per line.
int set_partition(CHPlan* p, int P) {
  Lines L;
  int rc = make_lines(p->n, P, p->a, p->noflux != 0, needs_scratch(p->n, P) ? p->n : 0, &L);
  if (rc != CS_OK) return rc;
  drop_graphs(p);
  free_lines(&p->lines);
  p->lines = L;
  p->P = P;
  p->m = static_cast<int>(p->n / P);
  return CS_OK;
}

}  // namespace

// Times one step for the plan's chunk count and every power of two (1 .. 64 chunks per line) from the plan's current
// state, keeps the fastest, records it in the tuning table, and restores the fields.
int ch_autotune(CHPlan* p, cudaStream_t s) {
  const size_t eb = p->storage == CS_F32 ? 4 : 8;
  const size_t bytes = static_cast<size_t>(p->n) * p->n * eb;
  void* save[2] = {nullptr, nullptr};
  CS_CUDA_TRY(cudaMalloc(&save[0], bytes));
  cudaError_t e = cudaMalloc(&save[1], bytes);
  if (e != cudaSuccess) { cudaFree(save[0]); return cuda_error(e, "autotune state copy"); }
  const int ip = p->iprev, ic = p->icur, in = p->inext;
  const int64_t steps = p->steps;
  e = cudaMemcpyAsync(save[0], p->field[ip], bytes, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(save[1], p->field[ic], bytes, cudaMemcpyDeviceToDevice, s);
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (e == cudaSuccess) e = cudaEventCreate(&e0);
  if (e == cudaSuccess) e = cudaEventCreate(&e1);
  int rc = e == cudaSuccess ? CS_OK : cuda_error(e, "autotune setup");
  int best = p->P;
  float best_ms = 1e30f;
  const int first = p->P;  // the plan's own partition first: another has to beat it
  for (int c = 0; c <= 7 && rc == CS_OK; ++c) {
    const int P = c == 0 ? first : 1 << (c - 1);
    if (!valid_chunks(p->n, P) || (c > 0 && P == first)) continue;
    rc = set_partition(p, P);
    if (rc != CS_OK) break;
    rc = ch_step(p, 1, nullptr, nullptr, s);  // warm-up
    if (rc != CS_OK) break;
    cudaEventRecord(e0, s);
    rc = ch_step(p, 2, nullptr, nullptr, s);
    cudaEventRecord(e1, s);
    if (rc != CS_OK) break;
    e = cudaEventSynchronize(e1);
    if (e != cudaSuccess) { rc = cuda_error(e, "autotune timing"); break; }
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    if (ms < best_ms) { best_ms = ms; best = P; }
  }
  if (rc == CS_OK) rc = set_partition(p, best);
  // restore the state the caller had
  p->iprev = ip; p->icur = ic; p->inext = in; p->steps = steps;
  cudaMemcpyAsync(p->field[ip], save[0], bytes, cudaMemcpyDeviceToDevice, s);
  cudaMemcpyAsync(p->field[ic], save[1], bytes, cudaMemcpyDeviceToDevice, s);
  cudaStreamSynchronize(s);
  cudaFree(save[0]); cudaFree(save[1]);
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  if (rc != CS_OK) return rc;
  tune_store(partition_key(p->storage, p->noflux, p->n), best);
  return CS_OK;
}

int ch_set_fields(CHPlan* p, void* prev, void* cur, void* next) {
  if (!prev || !cur || !next) return set_error(CS_EINVAL, "null field buffer");
  const size_t eb = p->storage == CS_F32 ? 4 : 8;
  const size_t bytes = static_cast<size_t>(p->n) * p->n * eb;
  void* f[3] = {prev, cur, next};
  for (int i = 0; i < 3; ++i) {
    if (reinterpret_cast<uintptr_t>(f[i]) % eb) return set_error(CS_EINVAL, "fields must be aligned to the element size");
    for (int j = i + 1; j < 3; ++j) {
      const char* a = static_cast<const char*>(f[i]);
      const char* b = static_cast<const char*>(f[j]);
      if (a < b + bytes && b < a + bytes) return set_error(CS_EALIAS, "the three fields must not overlap");
    }
  }
  drop_graphs(p);
  p->field[0] = prev; p->field[1] = cur; p->field[2] = next;
  p->iprev = 0; p->icur = 1; p->inext = 2;
  p->steps = 0;
  return CS_OK;
}

int ch_config(CHPlan* p, int32_t* chunks, int32_t* chunk_len) {
  if (chunks) *chunks = p->P;
  if (chunk_len) *chunk_len = p->m;
  return CS_OK;
}

void ch_destroy(CHPlan* p) { free_plan(p); }

// ---- a row band of a grid decomposed over several GPUs ----------------------------------------------
// The pieces of the ADI step that a caller runs on its own band of rows (Sec. 6.2's decomposition),
// periodic or with no-flux boundaries:
// the right-hand side and invariant sums of the band from padded C^n, C^{n-1} (2 halo rows each
// side, exchanged by the caller), line solves along the rows of a buffer (the x lines of the band,
// or after a transpose the y lines of a band of columns), and the update C^{n+1} = Cbar + v on the
// band.  The kernels are the full-grid step's own, so the decomposed step gives the same values.
struct CHBand {
  int64_t n, rows;
  int storage;
  int noflux;  // CS_CH_NOFLUX: mirrored columns, non-cyclic line solves
  double D, gamma, dt, h, a, alpha;
  int P, m;
  Lines lines;       // scratch for n lines: the band's columns, or its rows
  double* B;         // rows * n scratch (the local solutions of the columns, or of rows that do not fit in shared memory)
  double* partials;  // 2 per RHS block
  int rhs_blocks;
};

namespace {
template <typename T>
__global__ void __launch_bounds__(256)
    k_ch_band_update(const T* __restrict__ prev, const T* __restrict__ cur, const double* __restrict__ v,
                     T* __restrict__ next, int64_t n, int64_t count) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const int64_t o = i + 2 * n;  // padded row r + 2
  if constexpr (sizeof(T) == 4) {
    const float cb = fmaf(2.0f, cur[o], -prev[o]);  // as the full-grid update forms it
    next[o] = narrow_rn(widen(cb) + v[i]);
  } else {
    next[o] = fma(2.0, cur[o], -prev[o]) + v[i];
  }
}

void free_band(CHBand* b) {
  if (!b) return;
  free_lines(&b->lines);
  cudaFree(b->B); cudaFree(b->partials);
  delete b;
}
}  // namespace

// The partition (chunks per line) cs_ch_create picks for a description: the autotuner's choice
// for it when one is recorded, else the default.
static int band_partition(const cs_ch_desc* d) {
  int P = default_chunks(d->n), choice;
  if (tune_lookup(partition_key(d->storage, d->boundary == CS_CH_NOFLUX, d->n), &choice) && valid_chunks(d->n, choice)) P = choice;
  return P;
}

int ch_band_create(CHBand** out, const cs_ch_desc* d, int64_t rows) {
  *out = nullptr;
  if (!d) return set_error(CS_EINVAL, "null Cahn-Hilliard description");
  if (d->boundary != CS_CH_PERIODIC && d->boundary != CS_CH_NOFLUX)
    return set_error(CS_EINVAL, "boundary must be CS_CH_PERIODIC or CS_CH_NOFLUX");
  if (d->n < 64 || d->n % 64 != 0 || d->n > 65536) return set_error(CS_EINVAL, "n must be a multiple of 64 in [64, 65536]");
  if (rows < kTY || rows % kTY != 0 || rows > d->n) return set_error(CS_EINVAL, "band rows must be a multiple of %d in [%d, n]", kTY, kTY);
  if (d->storage != CS_F64 && d->storage != CS_F32) return set_error(CS_EINVAL, "storage must be CS_F64 or CS_F32");
  if (!(d->D > 0) || !(d->gamma >= 0) || !(d->dt > 0) || !std::isfinite(d->D) || !std::isfinite(d->gamma) || !std::isfinite(d->dt))
    return set_error(CS_EINVAL, "D > 0, gamma >= 0, dt > 0 and finite are required");
  CHBand* b = new (std::nothrow) CHBand;
  if (!b) return set_error(CS_ENOMEM, "out of host memory");
  memset(b, 0, sizeof *b);
  b->n = d->n; b->rows = rows; b->storage = d->storage;
  b->noflux = d->boundary == CS_CH_NOFLUX;
  b->D = d->D; b->gamma = d->gamma; b->dt = d->dt;
  b->h = 2.0 * M_PI / static_cast<double>(d->n);
  const double h2 = b->h * b->h;
  b->a = (2.0 / 3.0) * d->D * d->gamma * d->dt / (h2 * h2);
  b->alpha = (2.0 / 3.0) * d->D * d->dt / h2;
  const int P = band_partition(d);  // the full-grid plan's partition
  b->P = P;
  b->m = static_cast<int>(d->n / P);
  b->rhs_blocks = static_cast<int>((d->n / kTX) * (rows / kTY));
  int rc = make_lines(d->n, P, b->a, b->noflux != 0, d->n, &b->lines);
  if (rc != CS_OK) { free_band(b); return rc; }
  cudaError_t e = cudaMalloc(&b->B, static_cast<size_t>(rows) * d->n * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&b->partials, static_cast<size_t>(2) * b->rhs_blocks * sizeof(double));
  if (e != cudaSuccess) {
    free_band(b);
    return e == cudaErrorMemoryAllocation ? set_error(CS_ENOMEM, "band workspace: %s", cudaGetErrorString(e))
                                          : cuda_error(e, "band workspace");
  }
  rc = d->storage == CS_F32 ? set_rhs_attr<float>() : set_rhs_attr<double>();
  if (rc == CS_OK) rc = set_line_attrs();
  if (rc != CS_OK) { free_band(b); return rc; }
  *out = b;
  return CS_OK;
}

int ch_band_rhs(CHBand* b, const void* prev, const void* cur, double* rhs, double* sums, cudaStream_t s) {
  if (!prev || !cur || (!rhs && !sums)) return set_error(CS_EINVAL, "null buffer");
  dim3 grid(static_cast<unsigned>(b->n / kTX), static_cast<unsigned>(b->rows / kTY));
  const double hg = 0.5 * b->gamma / (b->h * b->h);
  double* part = sums ? b->partials : nullptr;
  if (b->storage == CS_F32)
    k_ch_rhs<float><<<grid, kThreads, rhs_smem_bytes(), s>>>(static_cast<const float*>(cur), static_cast<const float*>(prev),
                                                              rhs, b->n, b->alpha, b->a, hg, part, b->noflux,
                                                              ixd::ixi_round51(-b->a),
                                                              cubic_inv(b->alpha, ixd::ixi_round51(-b->a)), 1, nullptr);
  else
    k_ch_rhs<double><<<grid, kThreads, rhs_smem_bytes(), s>>>(static_cast<const double*>(cur), static_cast<const double*>(prev),
                                                               rhs, b->n, b->alpha, b->a, hg, part, b->noflux,
                                                               ixd::ixi_round51(-b->a),
                                                               cubic_inv(b->alpha, ixd::ixi_round51(-b->a)), 1, nullptr);
  CS_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  if (sums) {
    k_reduce_final<<<1, 256, 0, s>>>(b->partials, b->rhs_blocks, b->h * b->h, sums);
    CS_CUDA_TRY(cudaGetLastError());
    count_launches(1);
  }
  return CS_OK;
}

int ch_band_solve(CHBand* b, const double* in, double* out, cudaStream_t s) {
  if (!in || !out) return set_error(CS_EINVAL, "null buffer");
  // rows lines of n points
  return launch_rows(b->lines, b->noflux != 0, b->rows, in, out, b->B, s);
}

int ch_partition(const cs_ch_desc* d, int32_t* chunks, int32_t* chunk_len) {
  if (!d) return set_error(CS_EINVAL, "null Cahn-Hilliard description");
  if (d->n < 64 || d->n % 64 != 0 || d->n > 65536) return set_error(CS_EINVAL, "n must be a multiple of 64 in [64, 65536]");
  if (d->boundary != CS_CH_PERIODIC && d->boundary != CS_CH_NOFLUX)
    return set_error(CS_EINVAL, "boundary must be CS_CH_PERIODIC or CS_CH_NOFLUX");
  const int P = band_partition(d);
  if (chunks) *chunks = P;
  if (chunk_len) *chunk_len = static_cast<int32_t>(d->n / P);
  return CS_OK;
}

// The y lines of a band whose rows are whole chunks of those lines: chunks chunk0 .. chunk0 +
// rows / m - 1 of every column.  Phase 1 solves each of them locally (the x pass's own kernel with
// lines = the n columns, line stride 1, element stride n) into the plan's scratch and writes their
// end values to ends; phase 2, once the caller has gathered every band's end values in chunk order,
// applies the spike correction and writes v.
static int band_ycols_check(const CHBand* b, int64_t chunk0) {
  if (b->rows % b->m != 0)
    return set_error(CS_EINVAL, "band of %lld rows is not a whole number of %d-row chunks", (long long)b->rows, b->m);
  if (chunk0 < 0 || chunk0 + b->rows / b->m > b->P)
    return set_error(CS_EINVAL, "chunks %lld .. %lld outside the %d chunks of a line", (long long)chunk0,
                     (long long)(chunk0 + b->rows / b->m - 1), b->P);
  return CS_OK;
}

int ch_band_ycols_local(CHBand* b, int64_t chunk0, const double* in, double* ends, cudaStream_t s) {
  if (!in || !ends) return set_error(CS_EINVAL, "null buffer");
  int rc = band_ycols_check(b, chunk0);
  if (rc != CS_OK) return rc;
  const int Pl = static_cast<int>(b->rows / b->m);
  const unsigned sgrid = static_cast<unsigned>((b->n * Pl + kSolveThreads - 1) / kSolveThreads);
  k_line_local<AccStride><<<sgrid, kSolveThreads, 0, s>>>(in, reinterpret_cast<uint64_t*>(b->B), ends, line_scale(b->lines, b->n),
                                               b->lines.par, b->n, Pl, b->m, 1, b->n);
  CS_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  return CS_OK;
}

int ch_band_ycols_correct(CHBand* b, int64_t chunk0, const double* ends_all, double* v, cudaStream_t s) {
  if (!ends_all || !v) return set_error(CS_EINVAL, "null buffer");
  int rc = band_ycols_check(b, chunk0);
  if (rc != CS_OK) return rc;
  const int Pl = static_cast<int>(b->rows / b->m);
  const unsigned sgrid = static_cast<unsigned>((b->n * Pl + kSolveThreads - 1) / kSolveThreads);
  launch_states(b->lines, b->noflux != 0, b->n, ends_all, s);
  k_line_correct<0, double><<<sgrid, kSolveThreads, 0, s>>>(
      reinterpret_cast<uint64_t*>(b->B), line_states(b->lines, b->n), line_scale(b->lines, b->n), b->lines.par,
      line_tab(b->lines), b->n, static_cast<int>(chunk0), Pl, b->m, 1, b->n, v, static_cast<double*>(nullptr));
  CS_CUDA_TRY(cudaGetLastError());
  count_launches(2);
  return CS_OK;
}

int ch_band_update(CHBand* b, const void* prev, const void* cur, const double* v, void* next, cudaStream_t s) {
  if (!prev || !cur || !v || !next) return set_error(CS_EINVAL, "null buffer");
  const int64_t count = b->rows * b->n;
  const unsigned grid = static_cast<unsigned>((count + 255) / 256);
  if (b->storage == CS_F32)
    k_ch_band_update<float><<<grid, 256, 0, s>>>(static_cast<const float*>(prev), static_cast<const float*>(cur), v,
                                                 static_cast<float*>(next), b->n, count);
  else
    k_ch_band_update<double><<<grid, 256, 0, s>>>(static_cast<const double*>(prev), static_cast<const double*>(cur), v,
                                                  static_cast<double*>(next), b->n, count);
  CS_CUDA_TRY(cudaGetLastError());
  count_launches(1);
  return CS_OK;
}

void ch_band_destroy(CHBand* b) { free_band(b); }

// Host replay of the device line solver (the kernels' own functions, in their order) on the tables
// cs_ch_create builds, for a pseudo-random right-hand side; returns the backward error ||L x - b||_inf / ((1 + 16 a) ||x||_inf) of the result against the line operator
// itself (periodic: circulant (1, -4, 6, -4, 1); no-flux: reflected rows at the ends).
int ch_solver_check(int64_t n, int P, double a, bool noflux, double* residual) {
  if (!residual) return set_error(CS_EINVAL, "null residual pointer");
  if (n < 16 || n > 65536 || !valid_chunks(n, P)) return set_error(CS_EINVAL, "invalid line length / chunk count");
  if (!(a >= 0.0) || !std::isfinite(a)) return set_error(CS_EINVAL, "a must be finite and >= 0");
  pn::Par q;
  std::vector<pn::TabRow> tab;
  std::vector<uint64_t> base;
  std::vector<double> mats;
  if (!pn::build(n, P, a, noflux, q, tab, base, mats)) return set_error(CS_EINVAL, "a = %g is outside the solver's range", a);
  std::vector<double> b(n), x(n);
  uint64_t st = 0x9E3779B97F4A7C15ull ^ static_cast<uint64_t>(n * 131 + P);
  for (int64_t i = 0; i < n; ++i) {  // xorshift64*: values in [-1, 1)
    st ^= st >> 12; st ^= st << 25; st ^= st >> 27;
    b[i] = static_cast<double>((st * 0x2545F4914F6CDD1Dull) >> 11) * 0x1p-52 - 1.0;
  }
  pn::solve_host(q, tab, base, mats, n, P, noflux, b.data(), x.data());
  double rmax = 0.0, xmax = 0.0;
  auto at = [&](int64_t i) {  // periodic wrap or even reflection
    if (!noflux) return x[(i % n + n) % n];
    if (i < 0) i = -1 - i;
    if (i >= n) i = 2 * n - 1 - i;
    return x[i];
  };
  for (int64_t i = 0; i < n; ++i) {
    // L = I + a D4; D4 is the fourth difference, on the reflected line the square of the
    // reflected second difference, which reflection of x reproduces at every row
    double d2[3];
    for (int j = -1; j <= 1; ++j) d2[j + 1] = at(i + j - 1) - 2.0 * at(i + j) + at(i + j + 1);
    if (noflux) {  // D2 of the reflected line, taken again with reflection
      auto d2at = [&](int64_t k) {
        if (k < 0) k = -1 - k;
        if (k >= n) k = 2 * n - 1 - k;
        return at(k - 1) - 2.0 * at(k) + at(k + 1);
      };
      for (int j = -1; j <= 1; ++j) d2[j + 1] = d2at(i + j);
    }
    const double lx = x[i] + a * (d2[0] - 2.0 * d2[1] + d2[2]);
    rmax = std::max(rmax, std::fabs(lx - b[i]));
    xmax = std::max(xmax, std::fabs(x[i]));
  }
  *residual = rmax / ((1.0 + 16.0 * a) * std::max(xmax, 1e-300));
  return CS_OK;
}

}  // namespace cs
