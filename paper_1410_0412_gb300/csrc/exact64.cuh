// Integer-pipe arithmetic for the FP64 collision.
//
// GB300 executes FP64 arithmetic on two lanes per SM per clock, against 64
// integer and 128 FMA lanes, so an FP64 step written in FP64 instructions is
// bound by them while the other pipes idle.  The collision runs in 64-bit fixed
// point instead:
//
//  * the moments that the TRT collision (Sect. 2) starts from, the density
//    and momentum sums and the pair sums and differences: the 19 PDFs of a
//    node are converted to 64-bit fixed point with a per-node scale (the largest
//    exponent among them, with 5 bits of headroom) and summed exactly.  A PDF
//    at most 5 binades below the node's largest converts exactly; smaller ones
//    lose bits below 2^-57 of the largest.  Rounded once to the nearest double
//    (exact_moments), a moment's error is at most 19 * 2^-57 * max|f_i| plus
//    half an ulp of the result, below the error bound (n - 1) * 2^-53 * sum|f_i|
//    of the IEEE double sum of n terms that it replaces;
//  * the class terms and the pair update (FxClass, fx_class_int, fx_pairs),
//    rounded once per output;
//  * halving, where the FP64 update remains: an exponent decrement, identical
//    to 0.5 * x for every x whose half is a normal number, Inf or NaN.
//
// On the 256^3 bed (10.9 M nodes) the FP64 AA-R step pair went from 1.61 ms,
// with the class terms in FP64 (31 FP64 instructions a node), to 1.23 ms.  The even
// step of a 160^3 bed (3.03 M nodes, ncu): DRAM 77 %, integer pipe 66 %, FP64 pipe
// 67 %.
//
// All functions are __host__ __device__ so that a host test can check the
// moments bit for bit against exact rational arithmetic.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#include <cuda_runtime.h>

namespace lbm {
namespace dev {

__host__ __device__ __forceinline__ uint64_t dbits(double x) {
#ifdef __CUDA_ARCH__
  return static_cast<uint64_t>(__double_as_longlong(x));
#else
  uint64_t b;
  std::memcpy(&b, &x, sizeof b);
  return b;
#endif
}

__host__ __device__ __forceinline__ double dfrom(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(static_cast<long long>(b));
#else
  double x;
  std::memcpy(&x, &b, sizeof x);
  return x;
#endif
}

__host__ __device__ __forceinline__ int clz64(uint64_t a) {
#ifdef __CUDA_ARCH__
  return __clzll(static_cast<long long>(a));
#else
  return a ? __builtin_clzll(a) : 64;
#endif
}

constexpr uint64_t kSignBit = 0x8000000000000000ull;

// x / 2 without an FP64 instruction.  Exponent fields 2..2046 lose one; Inf and
// NaN pass through; zero, subnormals and the smallest binade shift their
// magnitude right (truncating the last subnormal bit).
__host__ __device__ __forceinline__ double halve_exact(double x) {
  const uint64_t b = dbits(x);
  const unsigned ef = static_cast<unsigned>(b >> 52) & 0x7ffu;
  uint64_t r;
  if (ef - 2u < 2045u)
    r = b - (uint64_t(1) << 52);
  else if (ef == 2047u)
    r = b;
  else
    r = (b & kSignBit) | ((b & ~kSignBit) >> 1);
  return dfrom(r);
}

// Smallest node scale: PDFs below 2^-959 (biased exponent 64) flush to zero.
constexpr int kFxMinExp = 64;
// Node scales at or above this biased exponent (|f| >= 2^1017) mark the node as
// diverged: the moments come out NaN, as an IEEE sum of such PDFs would.
constexpr int kFxMaxExp = 2040;

// Fixed-point image of the double with bits b at the node scale emax (the
// largest biased exponent among the node's PDFs, >= kFxMinExp):
// x * 2^(1080 - emax), truncated toward zero; |result| < 2^58.
__host__ __device__ __forceinline__ int64_t fx_of(uint64_t b, int emax) {
  const int e = static_cast<int>(b >> 52) & 0x7ff;
  const uint64_t m = ((b & 0x000fffffffffffffull) | 0x0010000000000000ull) << 10;  // < 2^63
  int sh = emax - e + 5;  // >= 5; zero and subnormal inputs (e = 0) shift out entirely
  sh = sh < 63 ? sh : 63;
  const uint64_t v = m >> sh;
  return (b & kSignBit) ? -static_cast<int64_t>(v) : static_cast<int64_t>(v);
}

// The double nearest to v * 2^(emax - 1080) (round to nearest, ties to even),
// for |v| < 2^63 and kFxMinExp <= emax < kFxMaxExp.
__host__ __device__ __forceinline__ double fx_to_double(int64_t v, int emax) {
  if (v == 0) return 0.0;
  const uint64_t s = static_cast<uint64_t>(v) & kSignBit;
  uint64_t a = v < 0 ? uint64_t(0) - static_cast<uint64_t>(v) : static_cast<uint64_t>(v);
  const int lz = clz64(a);  // >= 1
  a <<= lz;                 // leading one at bit 63
  uint64_t m = a >> 11;     // 53 significant bits
  const unsigned rest = static_cast<unsigned>(a) & 0x7ffu;
  m += (rest > 0x400u || (rest == 0x400u && (m & 1u))) ? 1u : 0u;
  // value = m * 2^(emax - lz - 1069); the biased exponent is emax + 6 - lz, and
  // adding m (hidden bit included, possibly 2^53 after rounding) to
  // (exponent - 1) << 52 assembles the bits with the carry in place.
  return dfrom(((static_cast<uint64_t>(emax + 5 - lz) << 52) + m) | s);
}

// 32-bit funnel shift (the PTX shf instruction) with a portable host image.
__host__ __device__ __forceinline__ uint32_t shf_l(uint32_t lo, uint32_t hi, unsigned n) {  // n in [0, 31]
#ifdef __CUDA_ARCH__
  return __funnelshift_l(lo, hi, n);
#else
  return n ? (hi << n) | (lo >> (32 - n)) : hi;
#endif
}

// fx_of for the common case, in 32-bit halves: a positive double (sign bit
// clear) at most 5 binades below the node's largest, so that fx_of's value
// m * 2^(10 - sh) is the significand m shifted left by k = 5 - (emax - e) in
// [0, 5].  Same value as fx_of (exact here).
__host__ __device__ __forceinline__ int64_t fx_of_pos_near(uint64_t b, unsigned k) {
  const uint32_t hi = static_cast<uint32_t>(b >> 32), lo = static_cast<uint32_t>(b);
  const uint32_t mh = (hi & 0x000fffffu) | 0x00100000u;  // significand bits 52..32, hidden bit included
  return static_cast<int64_t>((static_cast<uint64_t>(shf_l(lo, mh, k)) << 32) | (lo << k));
}

// fx_to_double through the hardware's int64 -> double conversion (round to
// nearest, ties to even: the same rounding, so the same bits), then an exact
// scaling by 2^(emax - 1080) as an exponent-field add.  The conversion is one
// instruction of the FP64 pipe, which has nothing else to do in the fixed-point
// collision (19 conversions a node keep it 60-70 % busy), and takes about 12
// instructions off the integer pipe, the busier one: with 9 / 7 / 5 of the
// pairs converted this way the FP64 AA-R pair on the 256^3 bed took 1.36 /
// 1.38 / 1.48 ms.  For kFxMinExp - 4 <= emax < kFxMaxExp every non-zero result
// is a normal number.
__host__ __device__ __forceinline__ double fx_to_double_cvt(int64_t v, int emax) {
#ifdef __CUDA_ARCH__
  const double x = __ll2double_rn(static_cast<long long>(v));
#else
  const double x = static_cast<double>(v);
#endif
  const uint64_t b = dbits(x);
  const uint32_t hi = static_cast<uint32_t>(b >> 32);
  const uint32_t scaled = hi ? hi + (static_cast<uint32_t>(emax - 1080) << 20) : 0u;
  return dfrom((static_cast<uint64_t>(scaled) << 32) | static_cast<uint32_t>(b));
}

// Node scale of the 19 PDFs: the largest biased exponent, at least emin (>= kFxMinExp).
template <int Q>
__host__ __device__ __forceinline__ int fx_scale(const uint64_t (&b)[Q], int emin = kFxMinExp) {
  int emax = emin;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int e = static_cast<int>(b[i] >> 52) & 0x7ff;
    emax = e > emax ? e : emax;
  }
  return emax;
}

// The exact fixed-point moments of one D3Q19 node from its 19 PDFs d (pair
// k = 1..9 holds the opposite directions 2k-1 and 2k; the first directions of
// the pairs are (1,0,0) (0,1,0) (0,0,1) (1,1,0) (1,-1,0) (1,0,1) (1,0,-1)
// (0,1,1) (0,1,-1)) at the node scale emax (returned): pair sums Sk[k] (only
// when NEED_SA) and differences D[k], the density deviation S = sum d_i and
// the momentum J = sum c_i d_i, all as integers times 2^(emax - 1080).
// FAST: the caller has checked fx_pos_near (positive PDFs within 5 binades
// of the largest) and passes the node scale it found as emax_fast; the
// conversions take the shorter fx_of_pos_near, and the integers are the same.
template <bool NEED_SA, bool FAST = false>
__host__ __device__ __forceinline__ int fx_moments(const double (&d)[19], int64_t (&Sk)[10], int64_t (&D)[10],
                                                   int64_t& S, int64_t& Jx, int64_t& Jy, int64_t& Jz,
                                                   int emax_fast = 0, int64_t* f0 = nullptr,
                                                   int emin = kFxMinExp) {
  uint64_t b[19];
#pragma unroll
  for (int i = 0; i < 19; ++i) b[i] = dbits(d[i]);
  int64_t f[19];
  int emax;
  if (FAST) {
    // positive: the exponent is the high word shifted, no sign to clear
    emax = emax_fast;
#pragma unroll
    for (int i = 0; i < 19; ++i) f[i] = fx_of_pos_near(b[i], static_cast<unsigned>(static_cast<int>(b[i] >> 52) + 5 - emax));
  } else {
    emax = fx_scale(b, emin);
#pragma unroll
    for (int i = 0; i < 19; ++i) f[i] = fx_of(b[i], emax);
  }
  S = f[0];
  if (f0) *f0 = f[0];
#pragma unroll
  for (int k = 1; k <= 9; ++k) {
    const int64_t s = f[2 * k - 1] + f[2 * k];
    D[k] = f[2 * k - 1] - f[2 * k];
    S += s;
    if (NEED_SA) Sk[k] = s;
  }
  Jx = D[1] + D[4] + D[5] + D[6] + D[7];
  Jy = D[2] + D[4] - D[5] + D[8] + D[9];
  Jz = D[3] + D[6] - D[7] + D[8] - D[9];
  return emax;
}

// Density deviation and momentum of single-precision PDFs as exact integers, in
// the terms of the doubles (scale 2^(emax - 1080), emax the returned double's
// biased exponent; kFxMaxExp for an Inf or a NaN).  Each PDF is split into three
// signed integers, x 2^(1080 - emax) = h 2^44 + l 2^22 + m with |h| <= 2^14 and
// |l|, |m| <= 2^21, by adding and subtracting 1.5 2^23 (every step but the last
// rounding is exact): eight instructions of the FMA pipe, which has nothing
// else to do here, instead of about eleven of the integer pipe, and 32-bit sums
// per slice instead of 64-bit ones.  Exact for PDFs within 34 binades of the
// largest.  Read-back of 5.3 M FP32 nodes: 410 us by shifts, 404 so.
__host__ __device__ __forceinline__ uint32_t fbits(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  uint32_t b;
  std::memcpy(&b, &x, sizeof b);
  return b;
#endif
}
__host__ __device__ __forceinline__ float ffrom(uint32_t b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float x;
  std::memcpy(&x, &b, sizeof x);
  return x;
#endif
}
__host__ __device__ __forceinline__ int fx_moments(const float (&d)[19], int64_t& S, int64_t& Jx, int64_t& Jy,
                                                   int64_t& Jz) {
  uint32_t top = 13u << 23;
#pragma unroll
  for (int i = 0; i < 19; ++i) {
    const uint32_t m = fbits(d[i]) & 0x7fffffffu;
    top = m > top ? m : top;
  }
  const float up = ffrom((267u - (top >> 23 < 254u ? top >> 23 : 254u)) << 23);  // 2^(140 - E): |x| up < 2^14
  constexpr float kM = 12582912.0f;                                              // 1.5 2^23
  constexpr uint32_t kMBits = 0x4b400000u;
  uint32_t h[19], l[19], m[19];
#pragma unroll
  for (int i = 0; i < 19; ++i) {
    const float s = d[i] * up;
    const float a = s + kM, r = s - (a - kM);
    const float b = std::fma(r, 4194304.0f, kM), q = std::fma(r, 4194304.0f, kM - b);
    h[i] = fbits(a);
    l[i] = fbits(b);
    m[i] = fbits(std::fma(q, 4194304.0f, kM));
  }
  auto join = [](uint32_t a, uint32_t b, uint32_t c) {
    return static_cast<int64_t>(static_cast<int32_t>(a)) * (int64_t(1) << 44) +
           static_cast<int64_t>(static_cast<int32_t>(b)) * (int64_t(1) << 22) + static_cast<int32_t>(c);
  };
  uint32_t s3[3], x3[3], y3[3], z3[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const uint32_t(&v)[19] = k == 0 ? h : k == 1 ? l : m;
    uint32_t t = v[0] - 19u * kMBits, D[10];
#pragma unroll
    for (int p = 1; p <= 9; ++p) {
      t += v[2 * p - 1] + v[2 * p];
      D[p] = v[2 * p - 1] - v[2 * p];
    }
    s3[k] = t;
    x3[k] = D[1] + D[4] + D[5] + D[6] + D[7];
    y3[k] = D[2] + D[4] - D[5] + D[8] + D[9];
    z3[k] = D[3] + D[6] - D[7] + D[8] - D[9];
  }
  S = join(s3[0], s3[1], s3[2]);
  Jx = join(x3[0], x3[1], x3[2]);
  Jy = join(y3[0], y3[1], y3[2]);
  Jz = join(z3[0], z3[1], z3[2]);
  return top >= 0x7f800000u ? kFxMaxExp : static_cast<int>(top >> 23) + 896;
}
__host__ __device__ __forceinline__ int fx_moments(const double (&d)[19], int64_t& S, int64_t& Jx, int64_t& Jy,
                                                   int64_t& Jz) {
  int64_t Sk[10], D[10];
  return fx_moments<false>(d, Sk, D, S, Jx, Jy, Jz);
}

// True when the fast conversions of fx_moments apply: every PDF positive and
// finite-scaled (node scale below kFxMaxExp) and at most 5 binades below the
// largest (so fx_of_pos_near's shift stays in [0, 5]; PDFs near w_i rho span
// 4).  emax: the node scale (the largest exponent field; meaningful when true).
__host__ __device__ __forceinline__ bool fx_pos_near(const double (&d)[19], int& emax) {
  // positive doubles order like their high words, and one negative high word
  // makes the minimum negative: a min and a max per PDF decide
  int32_t mn = 0x7fffffff, mx = 0;
#pragma unroll
  for (int i = 0; i < 19; ++i) {
    const int32_t hi = static_cast<int32_t>(dbits(d[i]) >> 32);
    mn = hi < mn ? hi : mn;
    mx = hi > mx ? hi : mx;
  }
  emax = mx >> 20;
  return (mn >> 20) >= kFxMinExp && emax < kFxMaxExp && emax - (mn >> 20) <= 5;
}

// The moments as doubles (lbm_exact_moments_host; the kernels keep the integers):
// pair sums sa_k (only when NEED_SA) and differences
// da_k, the density deviation drho = sum d_i and the momentum j = sum c_i d_i,
// each the double nearest to the exact fixed-point sum.  A node whose scale
// reaches kFxMaxExp (an Inf, a NaN or |d_i| >= 2^1017) gets drho = NaN.
template <bool NEED_SA>
__host__ __device__ __forceinline__ void exact_moments(const double (&d)[19], double (&sa)[10], double (&da)[10],
                                                       double& drho, double& jx, double& jy, double& jz) {
  int64_t Sk[10], D[10], S, Jx, Jy, Jz;
  const int emax = fx_moments<NEED_SA>(d, Sk, D, S, Jx, Jy, Jz);
#pragma unroll
  for (int k = 1; k <= 9; ++k) {
    if (NEED_SA) sa[k] = fx_to_double(Sk[k], emax);
    da[k] = fx_to_double(D[k], emax);
  }
  drho = emax < kFxMaxExp ? fx_to_double(S, emax) : dfrom(0x7ff8000000000000ull);
  jx = fx_to_double(Jx, emax);
  jy = fx_to_double(Jy, emax);
  jz = fx_to_double(Jz, emax);
}

// a * b / 2^64 for signed 64-bit a, b, within 3/4 of a unit (unbiased): the
// product of a Q64 fraction (|a| < 2^63, the value a / 2^64) with a fixed-point
// value, at the latter's scale.  Both factors are split in balanced halves
// (a = ah 2^32 + al with al a signed 32-bit word), so every partial product is
// one signed 32 x 32 -> 64 multiply-add on the FMA pipe, and the product of
// the low words, at most a quarter of a unit, is left out: three multiply-adds
// and about four ALU instructions, where the exact high word of a signed
// 64 x 64 product takes about 14.  Both factors must stay below 2^63 - 2^31
// in magnitude: the high halves, which round up, are then below 2^31 and the
// middle sum below 2^63.
struct Bal {
  int32_t h, l;
};
__host__ __device__ __forceinline__ Bal bal(int64_t v) {
  const int32_t l = static_cast<int32_t>(v);
  return Bal{static_cast<int32_t>(v >> 32) + static_cast<int32_t>(static_cast<uint32_t>(l) >> 31), l};
}
__host__ __device__ __forceinline__ int64_t mulhi_q64(Bal a, Bal b) {
  int64_t m = static_cast<int64_t>(a.h) * b.l + 0x80000000ll;
  m += static_cast<int64_t>(b.h) * a.l;
  return static_cast<int64_t>(a.h) * b.h + (m >> 32);
}
__host__ __device__ __forceinline__ int64_t mulhi_q64(int64_t a, int64_t b) { return mulhi_q64(bal(a), bal(b)); }

// Biased exponent field of a double.
__host__ __device__ __forceinline__ int dexp(double x) { return static_cast<int>(dbits(x) >> 52) & 0x7ff; }

// The pair update of the FP64 collision in fixed point (scale 2^(emax - 1080),
// the node's moment scale).  Given the class values of the TRT collision with
// Guo forcing -- the velocity u, the even constant K0 and the vectors T and O
// of the axis class (the diagonal class uses them halved) -- and the exact
// pair sums Sk and differences Dk, the post-collision pair is
//   e = K0 + (c.u)(c.T) [+ qp Sk],  o = qm Dk + c.O,  p_a = e + o,  p_b = e - o,
// with qm = (1 - l-)/2 and qp = (1 - l+)/2 as Q64 fractions.  The nine even
// products share six: (c.u)(c.T) is A_a = u_a T_a for an axis pair and
// A_a + A_b +- C_ab, C_ab = u_a T_b + u_b T_a, for a diagonal one.  The class
// values are held halved, as the six diagonal pairs use them.  The pair stage
// works at a scale kx bits finer than the moments, 2^(es - 1080) with
// es = emax - kx: Dk and Sk enter multiplied by 2^kx, exactly.  Every sum is
// exact; products are within 3/4 of a unit.  From class values given as
// doubles (fx_class, each truncated to the scale) the error of p before its
// one rounding to double is below 8 units of 2^(es - 1080), i.e. below
// 2^-(54 + kx) of B = 2^(emax - 1023), the binade of the node's largest PDF
// (for PDFs near w_i rho, below a quarter of an ulp of the smallest, the
// diagonal ones, when kx = 4).
//
// For class values given as doubles the host image takes kx = 4 when l+ = 1 and
// fx_room4, else 2; valid when |u_a| < 1/4 (biased exponent <= 1020), |K0| < B/2
// (exponent <= emax - 2) and |T_a|, |O_a| < B/4 (exponent <= emax - 3), which
// with every |d_i| < 2B keeps every intermediate below 2^63.  fx_class_ok
// checks it.
struct FxClass {
  int64_t K0;                 // even constant of the axis class
  int64_t Ax, Ay, Az;         // u_a T_a / 2
  int64_t Cxy, Cxz, Cyz;      // (u_a T_b + u_b T_a) / 2
  int64_t Ox, Oy, Oz;         // O_a / 2
};

// The even products from u (Q64) and T / 2.
__host__ __device__ __forceinline__ void fx_even(FxClass& q, int64_t ux, int64_t uy, int64_t uz, int64_t Tx, int64_t Ty,
                                                 int64_t Tz) {
  const Bal bx = bal(ux), by = bal(uy), bz = bal(uz), tx = bal(Tx), ty = bal(Ty), tz = bal(Tz);
  q.Ax = mulhi_q64(bx, tx);
  q.Ay = mulhi_q64(by, ty);
  q.Az = mulhi_q64(bz, tz);
  q.Cxy = mulhi_q64(bx, ty) + mulhi_q64(by, tx);
  q.Cxz = mulhi_q64(bx, tz) + mulhi_q64(bz, tx);
  q.Cyz = mulhi_q64(by, tz) + mulhi_q64(bz, ty);
}

__host__ __device__ __forceinline__ bool fx_class_ok(int emax, double ux, double uy, double uz, double K0, double Tx,
                                                     double Ty, double Tz, double Ox, double Oy, double Oz) {
  int eu = dexp(ux);
  eu = dexp(uy) > eu ? dexp(uy) : eu;
  eu = dexp(uz) > eu ? dexp(uz) : eu;
  int eto = dexp(Tx);
  const double v[5] = {Ty, Tz, Ox, Oy, Oz};
#pragma unroll
  for (int i = 0; i < 5; ++i) eto = dexp(v[i]) > eto ? dexp(v[i]) : eto;
  return emax < kFxMaxExp && eu <= 1020 && dexp(K0) <= emax - 2 && eto <= emax - 3;
}

// The bits of a value's high word that differ from its sign: fx_mag(v) < 2^k
// exactly when -2^(32 + k) <= v < 2^(32 + k).
__host__ __device__ __forceinline__ uint32_t fx_mag(int64_t v) {
  const int32_t h = static_cast<int32_t>(v >> 32);
  return static_cast<uint32_t>(h ^ (h >> 31));
}

// Whether the pair differences leave room for kx = 4: |D_k| 2^4 < 2^63 - 2^36 for
// mulhi_q64.  Only two PDFs of opposite signs, both within 2^-27 of 2^(emax - 1022),
// do not.
__host__ __device__ __forceinline__ bool fx_room4(const int64_t (&D)[10]) {
  uint32_t m = 0;
#pragma unroll
  for (int k = 1; k <= 9; ++k) m = fx_mag(D[k]) > m ? fx_mag(D[k]) : m;
  return m < (1u << 27) - 1;
}

// The class values at the pair scale es from doubles (see above).
__host__ __device__ __forceinline__ FxClass fx_class(int es, double ux, double uy, double uz, double K0, double Tx,
                                                     double Ty, double Tz, double Ox, double Oy, double Oz) {
  FxClass q;
  q.K0 = fx_of(dbits(K0), es);
  fx_even(q, fx_of(dbits(ux), 1016), fx_of(dbits(uy), 1016), fx_of(dbits(uz), 1016),  // u * 2^64
          fx_of(dbits(Tx), es + 1), fx_of(dbits(Ty), es + 1), fx_of(dbits(Tz), es + 1));
  q.Ox = fx_of(dbits(Ox), es + 1);
  q.Oy = fx_of(dbits(Oy), es + 1);
  q.Oz = fx_of(dbits(Oz), es + 1);
  return q;
}

// One pair from its even part e (without qp Sk) and c.O.  The two values are
// converted on the FP64 pipe (fx_to_double_cvt); GENERAL: with the integer
// routine, the same bits.
template <bool LP1, bool GENERAL>
__host__ __device__ __forceinline__ void fx_pair(int64_t e, int64_t co, int64_t Dk, int64_t Sk, Bal qm, Bal qp,
                                                 uint32_t px, int es, double& pa, double& pb) {
  // 2^kx D as a product: the FMA pipe has room, the integer pipe has not
  const int64_t o = mulhi_q64(qm, bal(static_cast<int64_t>(static_cast<uint64_t>(Dk) * px))) + co;
  if (!LP1) e += mulhi_q64(qp, bal(static_cast<int64_t>(static_cast<uint64_t>(Sk) * px)));
  pa = GENERAL ? fx_to_double(e + o, es) : fx_to_double_cvt(e + o, es);
  pb = GENERAL ? fx_to_double(e - o, es) : fx_to_double_cvt(e - o, es);
}

// The nine pairs in the direction order of the lattice (see fx_moments), from
// the moment-scale D and Sk of fx_moments; es = emax - kx.
template <bool LP1, bool GENERAL = false>
__host__ __device__ __forceinline__ void fx_pairs(const FxClass& q, const int64_t (&D)[10], const int64_t (&Sk)[10],
                                                  int64_t qm64, int64_t qp64, int es, int kx, double (&p)[19]) {
  const Bal qm = bal(qm64), qp = bal(qp64);
  const uint32_t px = 1u << kx;
  fx_pair<LP1, GENERAL>(q.K0 + 2 * q.Ax, 2 * q.Ox, D[1], Sk[1], qm, qp, px, es, p[1], p[2]);
  fx_pair<LP1, GENERAL>(q.K0 + 2 * q.Ay, 2 * q.Oy, D[2], Sk[2], qm, qp, px, es, p[3], p[4]);
  fx_pair<LP1, GENERAL>(q.K0 + 2 * q.Az, 2 * q.Oz, D[3], Sk[3], qm, qp, px, es, p[5], p[6]);
  const int64_t Kh = q.K0 >> 1;
  const int64_t Exy = Kh + q.Ax + q.Ay, Exz = Kh + q.Ax + q.Az, Eyz = Kh + q.Ay + q.Az;
  fx_pair<LP1, GENERAL>(Exy + q.Cxy, q.Ox + q.Oy, D[4], Sk[4], qm, qp, px, es, p[7], p[8]);
  fx_pair<LP1, GENERAL>(Exy - q.Cxy, q.Ox - q.Oy, D[5], Sk[5], qm, qp, px, es, p[9], p[10]);
  fx_pair<LP1, GENERAL>(Exz + q.Cxz, q.Ox + q.Oz, D[6], Sk[6], qm, qp, px, es, p[11], p[12]);
  fx_pair<LP1, GENERAL>(Exz - q.Cxz, q.Ox - q.Oz, D[7], Sk[7], qm, qp, px, es, p[13], p[14]);
  fx_pair<LP1, GENERAL>(Eyz + q.Cyz, q.Oy + q.Oz, D[8], Sk[8], qm, qp, px, es, p[15], p[16]);
  fx_pair<LP1, GENERAL>(Eyz - q.Cyz, q.Oy - q.Oz, D[9], Sk[9], qm, qp, px, es, p[17], p[18]);
}

// Q64 image of a rate constant |x| <= 1/2: round(x * 2^64), and whether mulhi_q64
// may take it: |x| 2^64 < 2^63 - 2^31.  A rate beyond that (1 - l+- within 2^-32 of
// +-1) has no image of its precision, and the caller takes the FP64 update.
inline bool q64_fits(double x) { return std::fabs(x) < 0.5 - 0x1p-33; }
inline int64_t q64_of(double x) { return q64_fits(x) ? static_cast<int64_t>(std::llround(std::ldexp(x, 64))) : 0; }

// ---- the class values in fixed point ---------------------------------------------------
//
// With exact integer moments S = sum d_i and J = sum c_i d_i, the class values
// of the pair update need no FP64 arithmetic either.  With q = rho u (which is
// kd (J + G/2), G = rho g, kd = 1 / (1 + s/2)) and F = G - s q, they are
//   T = K1 u + a+/2 F = l+/4 q + a+/2 F,   O = K2 u + a-/6 F = l-/6 q + a-/6 F,
//   K0 = l+/18 (S - 3/2 q.u) - 3 a+/18 u.F = l+/18 S - u.T / 3,
// all linear in q and F with per-launch Q64 constants; only u = q / rho, a
// factor of second-order products, takes a division (an integer reciprocal of
// rho, two Newton steps from a float estimate).  GB300 runs FP64 on 2 lanes
// per SM against 64 integer and 128 FMA lanes, and these terms in FP64 (27 to
// 50 instructions a node, 16 SM cycles a warp each) were what bound the FP64
// steps.
//
// The pair scale is 2^(es - 1080) with es = emax - kx: kx = 4 for full storage
// with l+ = 1, 2 for full storage otherwise, and 0 for deviations, whose momentum
// reaches 12 times their largest
// member.  Bounds (each checked, in units of the pair scale unless noted):
// |J_a| < 2^61, |G_a| < 2^59, |u_a| < 1/4, 0 <= s <= 1, and at the moment
// scale |S| < 2^60 (kx >= 2) or 2^62 (kx = 0, where also |S| >= 2^56 or some
// |J_a| >= 2^57).  With l+-, a+- in their ranges (k1 = l+/4 and a+/2 < 1/2,
// l-/6 < 1/3, a-/6 < 1/6) this gives |q| < 1.13
// 2^61, |F| < 1.38 2^61, |T| < 1.26 2^61, |c.T| < 2.51 2^61, |O| < 0.61 2^61,
// |K0| < 0.25 2^61 (0.45 2^61 at kx = 4) and every output below 2^63.
struct FxColl {
  int64_t k0a4;              // 4 l+/18 as a Q64 fraction, and so the next
  int64_t k1h, fsh;          // l+/8, a+/4 (T halved)
  int64_t k2h, foh;          // l-/12, a-/12 (O halved)
  int64_t qm, qp;            // (1 - l-)/2, (1 - l+)/2
  int64_t gm[3];             // body force: gm 2^(ge - 62), 2^62 <= |gm| < 2^63 (or 0)
  int ge[3];
  double rho_s;              // density of the storage shift, 0 for full storage
  bool shift;                // rho_s != 0 (a flag: the comparison is an FP64-pipe instruction)
  int emin;                  // least moment scale (deviation storage: that of the force)
  int emax;                  // moment scales from here on are out of range: kFxMaxExp, or 0 when a rate is (q64_fits)
  bool gx;                   // the force points along x
};

// The constants are the doubles of the FP64 update (make_coll), so that both
// updates evaluate the same map; those below 1/4 are exact as Q64 fractions.
inline FxColl make_fx_coll(double lp, double lm, const double (&g)[3], double rho_s) {
  FxColl c;
  const double ap = 1.0 - lp / 2, am = 1.0 - lm / 2;
  c.k0a4 = q64_of(4.0 * (lp / 18.0));
  c.k1h = q64_of(lp / 4.0 / 2.0);
  c.fsh = q64_of(ap / 2.0 / 2.0);
  c.k2h = q64_of(lm / 6.0 / 2.0);
  c.foh = q64_of(am / 6.0 / 2.0);
  c.qm = q64_of((1.0 - lm) / 2);
  c.qp = q64_of((1.0 - lp) / 2);
  c.emax = q64_fits((1.0 - lm) / 2) && q64_fits((1.0 - lp) / 2) ? kFxMaxExp : 0;
  for (int a = 0; a < 3; ++a) {
    int e = 0;
    const double m = std::frexp(g[a], &e);  // g = m 2^e, 1/2 <= |m| < 1
    c.gm[a] = static_cast<int64_t>(std::ldexp(m, 63));
    c.ge[a] = g[a] != 0.0 ? e - 1 : -4096;
  }
  c.rho_s = rho_s;
  c.shift = rho_s != 0.0;
  // deviations may be far below the force (a start from rest, strong drag):
  // the scale then follows rho g, the larger term of the result
  c.emin = kFxMinExp;
  if (rho_s != 0.0)
    for (int a = 0; a < 3; ++a) {
      const int e = dexp(rho_s * g[a]);
      c.emin = e > c.emin && e < kFxMaxExp ? e : c.emin;
    }
  c.gx = g[1] == 0.0 && g[2] == 0.0;
  return c;
}

__host__ __device__ __forceinline__ uint64_t umulhi64(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return static_cast<uint64_t>((static_cast<unsigned __int128>(a) * b) >> 64);
#endif
}

// 2^125 / D for 2^63 <= D < 2^64, within a relative 2^-60, in (2^61, 2^62]: a
// float estimate of the high word's reciprocal (21 bits or more) and two
// integer Newton steps.
__host__ __device__ __forceinline__ int64_t fx_recip(uint64_t D) {
  const uint32_t dh = static_cast<uint32_t>(D >> 32), dl = static_cast<uint32_t>(D);
  constexpr int64_t one = int64_t(1) << 62;
#ifdef __CUDA_ARCH__
  const uint32_t r0 = __float2uint_rz(__fdividef(4611686018427387904.0f, __uint2float_rz(dh)));  // 2^62 / dh
  const uint64_t low = __umulhi(dl, r0);
#else
  const uint32_t r0 = static_cast<uint32_t>(4611686018427387904.0f / static_cast<float>(dh));
  const uint64_t low = (static_cast<uint64_t>(dl) * r0) >> 32;
#endif
  const int64_t e = one - static_cast<int64_t>(static_cast<uint64_t>(dh) * r0 + low);  // |e| < 2^42
  const uint64_t r1 = (static_cast<uint64_t>(r0) << 32) +
                      static_cast<uint64_t>((static_cast<int64_t>(r0 >> 1) * static_cast<int32_t>(e >> 12)) >> 17);
  const int32_t e2 = static_cast<int32_t>(one - static_cast<int64_t>(umulhi64(D, r1)));
  return static_cast<int64_t>((r1 + static_cast<uint64_t>((static_cast<int64_t>(r1 >> 33) * e2) >> 29)) >> 1);
}

// Binades of the pair scale below the moments' (see above).  Uniform: a node's bits
// must not depend on the nodes that share its warp, and a scale chosen node by node
// costs the steps 1-2 %.
template <bool LP1> __host__ __device__ __forceinline__ int fx_kx(const FxColl& c) { return c.shift ? 0 : LP1 ? 4 : 2; }

// Class values at the pair scale of one node, from its moments at scale emax;
// false where a bound fails (the caller then takes the FP64 update).  s: the
// node's Brinkman solid fraction (DRAG only).
template <bool FORCE, bool DRAG, bool LP1>
__host__ __device__ __forceinline__ bool fx_class_int(const FxColl& c, int emax, int kx, int64_t S, int64_t Jx,
                                                      int64_t Jy, int64_t Jz, double s, FxClass& q) {
  const int es = emax - kx;
  // rho = D 2^(er - 63), 2^63 <= D < 2^64
  uint64_t D;
  int er;
  bool ok;
  if (c.shift) {  // uniform: deviation storage
    const uint64_t b = dbits(c.rho_s + fx_to_double_cvt(S, emax));
    D = (b << 11) | kSignBit;
    er = static_cast<int>(b >> 52) - 1023;  // a negative density, Inf or NaN: er >= 1024
    // |S| >= 2^56 or some |J_a| >= 2^57, unless the force sets the scale: where the
    // large deviations cancel in both, so do the results, and a scale tied to the
    // deviations would leave them few bits
    const uint32_t top = (fx_mag(S) << 1) | fx_mag(Jx) | fx_mag(Jy) | fx_mag(Jz);
    ok = er > -1000 && er < 1000 && fx_mag(S) < 1u << 30 && (top >= 1u << 25 || emax == c.emin);
  } else {
    const int lz = clz64(static_cast<uint64_t>(S));
    ok = S > 0 && fx_mag(S) < 1u << 28;
    D = (static_cast<uint64_t>(S) << (lz & 63)) | kSignBit;
    er = emax - 1017 - lz;
  }
  // u = q / rho will be mulhi(q 2^pre, r) 2^(3 - post), shifted left before
  // the product as far as |u| < 1/4 allows
  const int sh = es - 1016 - er;
  const int pre = sh > 1 ? sh - 1 : 0, down = 1 - sh + pre;  // >= 0
  const int post = down > 63 ? 63 : down;
  const int nj = (pre > 1 ? 30 - pre : 29) - kx;
  ok = ok && emax < c.emax && nj >= 0 && (fx_mag(Jx) | fx_mag(Jy) | fx_mag(Jz)) >> (nj & 31) == 0;
  const Bal r = bal(fx_recip(D));
  const uint32_t px = 1u << kx;
  int64_t qx = static_cast<int64_t>(static_cast<uint64_t>(Jx) * px);
  int64_t qy = static_cast<int64_t>(static_cast<uint64_t>(Jy) * px);
  int64_t qz = static_cast<int64_t>(static_cast<uint64_t>(Jz) * px);
  int64_t Fx = 0, Fy = 0, Fz = 0;
  if (FORCE || DRAG) {
    // rho g_a at the pair scale
    const Bal Dh = bal(static_cast<int64_t>(D >> 2));
    const int s0 = es - 1020 - er;
    const int shx = s0 - c.ge[0];
    ok = ok && shx >= 3 + pre;
    Fx = mulhi_q64(bal(c.gm[0] >> 1), Dh) >> (((shx > 65 ? 65 : shx) - 2) & 63);
    qx += Fx >> 1;
    if (!c.gx) {  // uniform
      const int shy = s0 - c.ge[1], shz = s0 - c.ge[2];
      ok = ok && shy >= 3 + pre && shz >= 3 + pre;
      Fy = mulhi_q64(bal(c.gm[1] >> 1), Dh) >> (((shy > 65 ? 65 : shy) - 2) & 63);
      Fz = mulhi_q64(bal(c.gm[2] >> 1), Dh) >> (((shz > 65 ? 65 : shz) - 2) & 63);
      qy += Fy >> 1;
      qz += Fz >> 1;
    }
  }
  if (DRAG) {
    const uint64_t b = dbits(s);
    ok = ok && b <= 0x3ff0000000000000ull;  // 0 <= s <= 1
    const int e = 1023 - static_cast<int>(b >> 52);
    // s/2 as a Q64 fraction (at most 2^63)
    const uint64_t sh2 = e < 64 ? (((b << 11) | kSignBit) >> (e & 63)) : 0u;
    const Bal kd = bal(fx_recip(kSignBit + (sh2 >> 1)));  // 1 / (1 + s/2), Q62
    qx = 2 * mulhi_q64(bal(2 * qx), kd);
    qy = 2 * mulhi_q64(bal(2 * qy), kd);
    qz = 2 * mulhi_q64(bal(2 * qz), kd);
    const Bal s4 = bal(static_cast<int64_t>(sh2 >> 1));
    Fx -= 2 * mulhi_q64(bal(2 * qx), s4);
    Fy -= 2 * mulhi_q64(bal(2 * qy), s4);
    Fz -= 2 * mulhi_q64(bal(2 * qz), s4);
  }
  const uint32_t pp = 1u << (pre & 31);
  auto velocity = [&](int64_t v) {
    const int64_t m = mulhi_q64(bal(static_cast<int64_t>(static_cast<uint64_t>(v) * pp)), r);
    return static_cast<int64_t>(static_cast<uint64_t>(m) << 3) >> post;
  };
  const int64_t ux = velocity(qx), uy = velocity(qy), uz = velocity(qz);
  ok = ok && (fx_mag(ux) | fx_mag(uy) | fx_mag(uz)) < 1u << 30;
  int64_t Tx, Ty, Tz;  // halved, as are Ox, Oy, Oz
  if (LP1) {  // l+/4 and a+/2 are both 1/4
    Tx = (qx + Fx) >> 3;
    Ty = (qy + Fy) >> 3;
    Tz = (qz + Fz) >> 3;
  } else {
    const Bal k1 = bal(c.k1h);
    Tx = mulhi_q64(k1, bal(qx));
    Ty = mulhi_q64(k1, bal(qy));
    Tz = mulhi_q64(k1, bal(qz));
  }
  const Bal k2 = bal(c.k2h);
  q.Ox = mulhi_q64(k2, bal(qx));
  q.Oy = mulhi_q64(k2, bal(qy));
  q.Oz = mulhi_q64(k2, bal(qz));
  if (FORCE || DRAG) {
    const Bal fs = bal(c.fsh), fo = bal(c.foh), fx = bal(Fx);
    q.Ox += mulhi_q64(fo, fx);
    if (!LP1) Tx += mulhi_q64(fs, fx);
    if (DRAG || !c.gx) {
      const Bal fy = bal(Fy), fz = bal(Fz);
      q.Oy += mulhi_q64(fo, fy);
      q.Oz += mulhi_q64(fo, fz);
      if (!LP1) {
        Ty += mulhi_q64(fs, fy);
        Tz += mulhi_q64(fs, fz);
      }
    }
  }
  fx_even(q, ux, uy, uz, Tx, Ty, Tz);
  // K0 = l+/18 S - u.T / 3
  const int64_t S2 = kx ? static_cast<int64_t>(static_cast<uint64_t>(S) << (kx - 2)) : S >> 2;
  constexpr int64_t third2 = 0x5555555555555555ll;  // 1/3 as a Q64 fraction
  q.K0 = mulhi_q64(c.k0a4, S2) - 2 * mulhi_q64(third2, q.Ax + q.Ay + q.Az);
  return ok;
}

// The post-collision PDFs of one node from its class values (fx_class_int),
// its moments at scale emax and the rest PDF's image f0.
template <bool LP1>
__host__ __device__ __forceinline__ void fx_update(const FxColl& c, const FxClass& q, int emax, int kx,
                                                   const int64_t (&D)[10], const int64_t (&Sk)[10], int64_t f0,
                                                   double (&d)[19]) {
  fx_pairs<LP1>(q, D, Sk, c.qm, c.qp, emax - kx, kx, d);
  // rest PDF: (1 - l+) f0 + 6 K0
  int64_t v0 = 6 * q.K0;
  if (!LP1) v0 += mulhi_q64(c.qp, static_cast<int64_t>(static_cast<uint64_t>(f0) << (kx + 1)));
  d[0] = fx_to_double_cvt(v0, emax - kx);
}

// J 2^(emax - 1080) / rho as a double within (1/2 + 2^-4) ulp, for |J| < 2^62
// (ten PDFs below 2^58), rho = D 2^(er - 63), 2^63 <= D < 2^64, r = fx_recip(D)
// and 64 <= emax - er < 1900.  J is shifted to 62 bits, so that the product keeps
// 58 or more.  Not to 63: mulhi_q64 takes factors below 2^63 - 2^31, and a J
// just below a power of two (a velocity of 1/16) came out with the wrong sign.
__host__ __device__ __forceinline__ double fx_quotient(int64_t J, int emax, Bal r, int er) {
  const uint64_t a = static_cast<uint64_t>(J ^ (J >> 63)) | 1u;
  const int lz = clz64(a);  // 2..63
  const int64_t m = mulhi_q64(bal(static_cast<int64_t>(static_cast<uint64_t>(J) << (lz - 2))), r);
  return fx_to_double_cvt(m, emax - er - lz + 4);  // m 2^(emax - er - lz - 1076)
}

// Density rho = rho_s + S and j / rho of one node from its moments (scale emax) by
// integer quotients; false for nodes outside their range (no positive normal
// density, Inf or NaN PDFs), whose quotients the caller forms in FP64.
__host__ __device__ __forceinline__ bool fx_velocity(double rho_s, int emax, int64_t S, int64_t Jx, int64_t Jy,
                                                     int64_t Jz, double& r, double& ux, double& uy, double& uz) {
  r = rho_s + fx_to_double_cvt(S, emax);
  const uint64_t b = dbits(r);
  const int er = static_cast<int>(b >> 52) - 1023;
  if (!(emax < kFxMaxExp && er > -1000 && er < 1000 && emax - er >= 64 && emax - er < 1900)) return false;
  const Bal q = bal(fx_recip((b << 11) | kSignBit));
  ux = fx_quotient(Jx, emax, q, er);
  uy = fx_quotient(Jy, emax, q, er);
  uz = fx_quotient(Jz, emax, q, er);
  return true;
}

// ---- the adjoint step in fixed point ----------------------------------------------------
//
// With the weighted moments M0, M1, M2 of the gathered adjoint vector mu and
// K = 9 M2 - 3 M0, the terms of the adjoint collision (adjoint.cu) collapse to
//   X = K u, Y = K g, P = dPsi/du = (l+ - 2 a+ s) X + a+ Y + 3 (l- - a- s) M1,
//   A = l+ M0 - (l+/2 - a+ s) u.X + 3 a- M1.g + kd P.g / 2,   B = kd P,
//   dJ/ds / rho = -a+ u.X - 3 a- M1.u - kd P.u / 2,
// all linear in mu: products of the integer moments (w = 1/36 and 1/18 make them
// integers over 36) with u, g and per-launch constants as Q64 fractions.  lambda is
// formed at mu's scale.  dJ/ds is a sum of products of M1, K, u and g, any of which
// may be small beside max|mu| or 1 (a smooth adjoint field, a slow flow), so each
// of the four is normalised first: K to K 2^zk and M1 to M1 2^zn (members below 2^62,
// the largest at 2^61 or more; K exactly, with the remainder of M0's third), u to u'
// 2^-p and g to g' 2^-zg with their largest components at 1/8 or more.  The three sums
// M1.u, u.X and Y.u keep 56 bits or more of their terms and are added in FP64.  At
// mu's scale throughout, dJ/ds lost 1e-12 of itself to rounding on a smooth field at
// |u| = 1e-6, where the FP64 form kept 1e-16.
//
// Bounds: |mu_i| < 2^58 at mu's scale, so |36 M0| / 2 < 18, |36 M1| < 12,
// |36 M2_aa| < 12, |36 M2_ab| < 4 and |4 K_aa| < 24 (times 2^58 each; normalised
// values below 16, or these at zk = zn = 0); |J 2^z| < 2^62, |G| < 2^59 and p >= 0
// give |u'| < 0.28 2^64 and |4 X| < 13.5 2^58; |g_a| < 2^-6 (checked on the host)
// makes Y small at mu's scale, and |g'| < 1/4 bounds it there; then |P| < 7 2^58,
// |A| < 5 2^58 and every output is below 2^62.  Each product is within 3/4 of a unit.
struct FxAdj {
  int64_t l18;           // l+/18 as a Q64 fraction, and so the next
  int64_t c1, c1s;       // l+/4, a+/2  (c1 - c1s s)
  int64_t c3, c3s;       // l-/12, a-/12 (c3 - c3s s)
  int64_t ap4;           // a+/4
  int64_t g[3], gn[3];   // g, and g 2^zg
  int zg;
  bool ok;               // the force and the rates are in range
};

inline FxAdj make_fx_adj(double lp, double lm, const double (&g)[3]) {
  FxAdj c;
  const double ap = 1.0 - lp / 2, am = 1.0 - lm / 2;
  c.l18 = q64_of(lp / 18.0);
  c.c1 = q64_of(lp / 4.0);
  c.c1s = q64_of(ap / 2.0);
  c.c3 = q64_of(lm / 12.0);
  c.c3s = q64_of(am / 12.0);
  c.ap4 = q64_of(ap / 4.0);
  c.ok = q64_fits(lp / 4.0) && q64_fits(ap / 2.0);
  double top = 0.0;
  for (int a = 0; a < 3; ++a) {
    c.ok = c.ok && std::fabs(g[a]) < 0.015625;
    top = std::fmax(top, std::fabs(g[a]));
  }
  int e = 0;
  std::frexp(top, &e);  // top in [2^(e - 1), 2^e)
  c.zg = c.ok && top > 0.0 ? -2 - e : 0;
  for (int a = 0; a < 3; ++a) {
    c.g[a] = c.ok ? q64_of(g[a]) : 0;
    c.gn[a] = c.ok ? q64_of(std::ldexp(g[a], c.zg)) : 0;
  }
  return c;
}

// Magnitude bits of a value, the shift that takes the largest of several (their bits
// or-ed) to [2^61, 2^62), at most 59 and 0 for larger ones, and shifts by such counts.
__host__ __device__ __forceinline__ uint64_t fx_bits(int64_t v) { return static_cast<uint64_t>(v ^ (v >> 63)); }
__host__ __device__ __forceinline__ int fx_norm(uint64_t bits) {
  const int n = clz64(bits) - 2;
  return n < 0 ? 0 : n > 59 ? 59 : n;
}
__host__ __device__ __forceinline__ int64_t fx_shl(int64_t v, int n) {
  return static_cast<int64_t>(static_cast<uint64_t>(v) << (n & 63));
}
__host__ __device__ __forceinline__ int64_t fx_shr(int64_t v, int n) { return v >> ((n > 63 ? 63 : n) & 63); }

// Least moment scale of the adjoint vector: leaves room below it for the finer
// scale of the gradient (adjoint values below 2^-880 flush to zero).
constexpr int kFxMinExpAdj = 200;

struct FxAdjOut {
  int64_t A, Bx, By, Bz;  // at mu's scale
  double gs;              // dJ/ds / rho
};

// A, B and the gradient term of one node: from the forward moments (S, J at
// scale ef) and the adjoint pair sums and differences Pi, Di and rest value m0 at
// scale em.  False where a bound fails (the caller takes the FP64 form).
template <bool DRAG>
__host__ __device__ __forceinline__ bool fx_adjoint(const FxColl& c, const FxAdj& a, int ef, int64_t S, int64_t Jx,
                                                    int64_t Jy, int64_t Jz, double s, int em, int64_t m0,
                                                    const int64_t (&Pi)[10], const int64_t (&Di)[10], FxAdjOut& o) {
  // rho = D 2^(er - 63)
  uint64_t D;
  int er;
  bool ok = a.ok && ef < c.emax && em < c.emax;
  if (c.shift) {  // uniform
    const uint64_t b = dbits(c.rho_s + fx_to_double_cvt(S, ef));
    D = (b << 11) | kSignBit;
    er = static_cast<int>(b >> 52) - 1023;
    ok = ok && er > -1000 && er < 1000;
  } else {
    const int lz = clz64(static_cast<uint64_t>(S));
    ok = ok && S > 0;
    D = (static_cast<uint64_t>(S) << (lz & 63)) | kSignBit;
    er = ef - 1017 - lz;
  }
  // q = rho u at z bits below the forward scale: J 2^z < 2^62, G < 2^59
  const uint64_t mj = static_cast<uint64_t>((Jx ^ (Jx >> 63)) | (Jy ^ (Jy >> 63)) | (Jz ^ (Jz >> 63)));
  int z = mj ? clz64(mj) - 2 : 4096;
  const int zg = ef - 1023 - er;
  z = zg - c.ge[0] < z ? zg - c.ge[0] : z;
  if (!c.gx) {  // uniform
    z = zg - c.ge[1] < z ? zg - c.ge[1] : z;
    z = zg - c.ge[2] < z ? zg - c.ge[2] : z;
  }
  ok = ok && z >= 0;
  const Bal Dh = bal(static_cast<int64_t>(D >> 2)), r = bal(fx_recip(D));
  const int s0 = ef - z - 1020 - er;
  const int shx = s0 - c.ge[0];
  int64_t qx = static_cast<int64_t>(static_cast<uint64_t>(Jx) << (z & 63)) +
               (mulhi_q64(bal(c.gm[0] >> 1), Dh) >> (((shx > 64 ? 64 : shx) - 1) & 63));
  int64_t qy = static_cast<int64_t>(static_cast<uint64_t>(Jy) << (z & 63));
  int64_t qz = static_cast<int64_t>(static_cast<uint64_t>(Jz) << (z & 63));
  if (!c.gx) {  // uniform
    const int shy = s0 - c.ge[1], shz = s0 - c.ge[2];
    qy += mulhi_q64(bal(c.gm[1] >> 1), Dh) >> (((shy > 64 ? 64 : shy) - 1) & 63);
    qz += mulhi_q64(bal(c.gm[2] >> 1), Dh) >> (((shz > 64 ? 64 : shz) - 1) & 63);
  }
  Bal kd = Bal{1 << 30, 0};  // Q62
  int64_t c1 = a.c1, c3 = a.c3;
  if (DRAG) {
    const uint64_t b = dbits(s);
    ok = ok && b <= 0x3ff0000000000000ull;  // 0 <= s <= 1
    const int e = 1023 - static_cast<int>(b >> 52);
    const uint64_t sh2 = e < 64 ? (((b << 11) | kSignBit) >> (e & 63)) : 0u;  // s/2, Q64
    kd = bal(fx_recip(kSignBit + (sh2 >> 1)));
    qx = 4 * mulhi_q64(bal(qx), kd);
    qy = 4 * mulhi_q64(bal(qy), kd);
    qz = 4 * mulhi_q64(bal(qz), kd);
    const Bal s4 = bal(static_cast<int64_t>(sh2 >> 1));  // s/4
    c1 -= 4 * mulhi_q64(bal(a.c1s), s4);
    c3 -= 4 * mulhi_q64(bal(a.c3s), s4);
  }
  // u' = mulhi(q, r) 2^(2 + ku), u = u' 2^-p (Q64), its largest component in [2^61, 2^62)
  const int64_t vx = 4 * mulhi_q64(bal(qx), r), vy = 4 * mulhi_q64(bal(qy), r), vz = 4 * mulhi_q64(bal(qz), r);
  const uint64_t mu = fx_bits(vx) | fx_bits(vy) | fx_bits(vz);
  const int ku = fx_norm(mu);
  const Bal ux = bal(fx_shl(vx, ku)), uy = bal(fx_shl(vy, ku)), uz = bal(fx_shl(vz, ku));
  const int p = (vx | vy | vz) != 0 ? z + ku + 1016 + er - ef : 0;
  ok = ok && p >= 0;
  // moments over 36 (M0 halved); 36 M0 = 3 t0 + rem, |rem| <= 6
  const int64_t A1 = Pi[1] + Pi[2] + Pi[3], Ad = Pi[4] + Pi[5] + Pi[6] + Pi[7] + Pi[8] + Pi[9];
  const int64_t m0h = 6 * m0 + A1 + (Ad >> 1);
  constexpr int64_t third = 0x5555555555555555ll;
  const int64_t t0 = 2 * mulhi_q64(third, m0h);
  const int64_t rem = static_cast<int64_t>(12 * static_cast<uint64_t>(m0) + 2 * static_cast<uint64_t>(A1) +
                                           static_cast<uint64_t>(Ad) - 3 * static_cast<uint64_t>(t0));
  // 4 K 2^zk and 36 M1 2^zn
  const int64_t lxx = 2 * Pi[1] + Pi[4] + Pi[5] + Pi[6] + Pi[7] - t0;
  const int64_t lyy = 2 * Pi[2] + Pi[4] + Pi[5] + Pi[8] + Pi[9] - t0;
  const int64_t lzz = 2 * Pi[3] + Pi[6] + Pi[7] + Pi[8] + Pi[9] - t0;
  const int64_t lxy = Pi[4] - Pi[5], lxz = Pi[6] - Pi[7], lyz = Pi[8] - Pi[9];
  const int zk = fx_norm(fx_bits(lxx) | fx_bits(lyy) | fx_bits(lzz) | fx_bits(lxy) | fx_bits(lxz) | fx_bits(lyz));
  const int64_t r3 = mulhi_q64(third, fx_shl(rem, zk));
  const Bal kxx = bal(fx_shl(lxx, zk) - r3), kyy = bal(fx_shl(lyy, zk) - r3), kzz = bal(fx_shl(lzz, zk) - r3);
  const Bal kxy = bal(fx_shl(lxy, zk)), kxz = bal(fx_shl(lxz, zk)), kyz = bal(fx_shl(lyz, zk));
  const int64_t hx = 2 * Di[1] + Di[4] + Di[5] + Di[6] + Di[7];
  const int64_t hy0 = 2 * Di[2] + Di[4] - Di[5] + Di[8] + Di[9];
  const int64_t hz = 2 * Di[3] + Di[6] - Di[7] + Di[8] - Di[9];
  const int zn = fx_norm(fx_bits(hx) | fx_bits(hy0) | fx_bits(hz));
  const Bal nx = bal(fx_shl(hx, zn)), ny = bal(fx_shl(hy0, zn)), nz = bal(fx_shl(hz, zn));
  // 4 X (scale em - p - zk), M1.u (36; em - p - zn) and 4 u.X (em - 2p - zk)
  const int64_t Xx = mulhi_q64(kxx, ux) + mulhi_q64(kxy, uy) + mulhi_q64(kxz, uz);
  const int64_t Xy = mulhi_q64(kxy, ux) + mulhi_q64(kyy, uy) + mulhi_q64(kyz, uz);
  const int64_t Xz = mulhi_q64(kxz, ux) + mulhi_q64(kyz, uy) + mulhi_q64(kzz, uz);
  const int64_t nu = mulhi_q64(nx, ux) + mulhi_q64(ny, uy) + mulhi_q64(nz, uz);
  const int64_t uX = mulhi_q64(ux, bal(Xx)) + mulhi_q64(uy, bal(Xy)) + mulhi_q64(uz, bal(Xz));
  // 4 Y (em - zk - zg), 4 Y.u (em - p - zk - zg) and M1.g (36; em - zn - zg)
  const Bal gx = bal(a.gn[0]);
  int64_t Yx = mulhi_q64(kxx, gx), Yy = mulhi_q64(kxy, gx), Yz = mulhi_q64(kxz, gx), ng = mulhi_q64(nx, gx);
  if (!c.gx) {  // uniform
    const Bal gy = bal(a.gn[1]), gz = bal(a.gn[2]);
    Yx += mulhi_q64(kxy, gy) + mulhi_q64(kxz, gz);
    Yy += mulhi_q64(kyy, gy) + mulhi_q64(kyz, gz);
    Yz += mulhi_q64(kyz, gy) + mulhi_q64(kzz, gz);
    ng += mulhi_q64(ny, gy) + mulhi_q64(nz, gz);
  }
  const int64_t uY = mulhi_q64(ux, bal(Yx)) + mulhi_q64(uy, bal(Yy)) + mulhi_q64(uz, bal(Yz));
  // back at mu's scale: P, M1.g and u.X
  const int sx = p + zk, sy = zk + a.zg;
  const Bal b1 = bal(c1), b3 = bal(c3), ap4 = bal(a.ap4);
  const int64_t Px = mulhi_q64(b1, bal(fx_shr(Xx, sx))) + mulhi_q64(ap4, bal(fx_shr(Yx, sy))) + fx_shr(mulhi_q64(b3, nx), zn);
  const int64_t Py = mulhi_q64(b1, bal(fx_shr(Xy, sx))) + mulhi_q64(ap4, bal(fx_shr(Yy, sy))) + fx_shr(mulhi_q64(b3, ny), zn);
  const int64_t Pz = mulhi_q64(b1, bal(fx_shr(Xz, sx))) + mulhi_q64(ap4, bal(fx_shr(Yz, sy))) + fx_shr(mulhi_q64(b3, nz), zn);
  int64_t Pg = mulhi_q64(bal(a.g[0]), bal(Px));
  if (!c.gx) Pg += mulhi_q64(bal(a.g[1]), bal(Py)) + mulhi_q64(bal(a.g[2]), bal(Pz));
  o.A = mulhi_q64(bal(a.l18), bal(m0h)) - (mulhi_q64(b1, bal(fx_shr(uX, sx + p))) >> 1) +
        mulhi_q64(bal(a.c3s), bal(fx_shr(ng, zn + a.zg)));
  if (DRAG) {
    o.A += 2 * mulhi_q64(kd, bal(Pg));
    o.Bx = 2 * mulhi_q64(kd, bal(2 * Px));
    o.By = 2 * mulhi_q64(kd, bal(2 * Py));
    o.Bz = 2 * mulhi_q64(kd, bal(2 * Pz));
  } else {
    o.A += Pg >> 1;
    o.Bx = Px;
    o.By = Py;
    o.Bz = Pz;
  }
  // -(a-/12 + kd/2 c3) M1.u - (a+/4 + kd/2 c1) u.X - kd/2 a+/4 u.Y
  const int64_t h3 = DRAG ? 2 * mulhi_q64(kd, b3) : c3 >> 1, h1 = DRAG ? 2 * mulhi_q64(kd, b1) : c1 >> 1;
  const int64_t hy = DRAG ? 2 * mulhi_q64(kd, ap4) : a.ap4 >> 1;
  // (the first factor below 1/12, the last below 1/8: times 4 and 2); terms below
  // 2^-948, of a velocity that small, flush to zero
  auto term = [](int64_t v, int e) { return e >= 70 ? fx_to_double_cvt(v, e) : 0.0; };
  const int en = em - p - zn, ex = em - p - sx, ey = em - p - sy;
  o.gs = -(term(mulhi_q64(bal(4 * (a.c3s + h3)), bal(nu)), en - 2) + term(mulhi_q64(bal(a.ap4 + h1), bal(uX)), ex) +
           term(mulhi_q64(bal(2 * hy), bal(uY)), ey - 1));
  return ok;
}

}  // namespace dev
}  // namespace lbm
