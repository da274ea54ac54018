// Multi-CTA class: haloes too large for one CTA's (or one cluster's) shared
// memory, and every halo in the all-FP64 mode.
//
// The haloes of this class share flat arrays (halo k owns [gbase_k,
// gbase_k + count_k)) cut into tiles of GRID_TILE elements that never cross
// a halo.  The steps are those of the on-chip classes (Sect. 2.1, Appendix
// A), laid out for HBM streaming:
//   prepare  one coalesced read of the candidates: recentring, sphere test,
//            radius key, and a 32-byte record per candidate, (w, r) and
//            (v, m) with w = v + H d (64 bytes in the all-FP64 mode)
//   sort     members distributed into radial bins by rank of arrival (counted
//            by the prepare), each bin then ordered on chip by one CTA, which
//            writes the radial-order streams (w, r), (v, 1/r), so no later step
//            touches the particle store.  Radii that the bins cannot hold
//            (thousands equal, a thin shell in a void) take a segmented stable LSD
//            radix sort of (key, position) with 8-bit digits instead
//   init     exact sums of the initial set per sub-tile (with the bins) and per
//            halo, v_bulk
//   passes   two kernels per iteration.  A streaming one: each sub-tile of an
//            active halo takes the exact prefix sums M(<r) and sum m/r of the
//            tiles before it from the tile prefixes of the current set,
//            evaluates phi (Appendix A), the escape test and the removals, and
//            subtracts what it removed from its own sums.  Then one CTA or warp
//            per halo (g_halo) turns the sub-tiles' sums into the prefixes of
//            the set left, the halo's totals, v_bulk, its convergence and its
//            part of the next pass's list
//   final    bound lists, phi, compacted radii and inclusive masses, the
//            first virial crossing, the records, and the profile rows by
//            binary search over the compacted radii
//
// No CTA ever waits for another one: a tile reads only prefixes that an
// earlier kernel finished.

// Exact sums: long long fixed point in the mixed mode (the same scales and
// bits as the on-chip classes), __int128 in the all-FP64 mode, where a
// 64-bit quantum would limit large haloes to ~1e-11 relative in sum m/r.
#include <algorithm>
#include <atomic>
#include <cstdint>

#include "ahf_device.cuh"

namespace ahf {
namespace {

constexpr int T = GRID_THREADS;         // 256
constexpr int TILE = GRID_TILE;         // 2048
constexpr int IPT = TILE / T;           // 8 elements per thread
constexpr int NWARP = T / 32;
static_assert(T == 256 && GRID_TILE == 2048, "one thread per byte digit in the histograms and scans");

// Precision of the per-particle arithmetic.  float: the mixed mode (FP32
// radius key, FP32 phi and escape test).  double: the all-FP64 mode (FP64
// offsets, radius key, phi and escape test).
struct alignas(32) D4 {
  double x, y, z, w;
};
template <typename R>
struct Prec;
template <>
struct Prec<float> {
  using Key = uint32_t;
  using V4 = float4;
  using Acc = long long;
  static constexpr int ACC_BITS = 61;   // partial sums stay below 2^62
};
template <>
struct Prec<double> {
  using Key = unsigned long long;
  using V4 = D4;
  using Acc = __int128;
  static constexpr int ACC_BITS = 125;  // partial sums stay below 2^126
};

// ---- exact sums ---------------------------------------------------------------------

template <typename Acc>
__device__ __forceinline__ Acc& A(AccSlot& s) {
  return *reinterpret_cast<Acc*>(s.w);
}
template <typename Acc>
__device__ __forceinline__ Acc Ald(const AccSlot& s) {
  return *reinterpret_cast<const Acc*>(s.w);
}
// an AccSlot another CTA of the running kernel wrote (read through L2)
template <typename Acc>
__device__ __forceinline__ Acc Acg(const AccSlot& s);
template <>
__device__ __forceinline__ long long Acg<long long>(const AccSlot& s) {
  return __ldcg(&s.w[0]);
}
template <>
__device__ __forceinline__ __int128 Acg<__int128>(const AccSlot& s) {
  const unsigned long long lo = (unsigned long long)__ldcg(&s.w[0]);
  const unsigned long long hi = (unsigned long long)__ldcg(&s.w[1]);
  return (__int128)(((unsigned __int128)hi << 64) | (unsigned __int128)lo);
}

// Scale exponent s for sums of n terms of magnitude < 2^(emax+1) (the mixed
// mode's is fix_scale's).
template <typename R>
__device__ __forceinline__ int acc_scale(int emax, long long n) {
  int bits = 0;
  while (bits < 40 && (1ll << bits) < n) ++bits;
  return Prec<R>::ACC_BITS - bits - emax;
}

// round(x 2^s) for the all-FP64 mode (round half away from zero); the caller
// guarantees |x| 2^s < 2^126.
__device__ __forceinline__ __int128 fix128_from_double(double x, int s) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff);
  if (e == 0) return 0;
  const long long mant = (long long)((b & 0xfffffffffffffull) | 0x10000000000000ull);
  const int sh = e - 1075 + s;
  __int128 v;
  if (sh >= 0) v = (__int128)mant << (sh > 73 ? 73 : sh);
  else if (sh > -54) v = (__int128)(((mant >> (-sh - 1)) + 1) >> 1);
  else v = 0;
  return (b >> 63) ? -v : v;
}

// v 2^-s as the nearest double (ties to even): the top 64 bits with every bit below
// ORed into the last, rounded to 53 by an add whose carry runs into the exponent.
// Integer instructions only: the FP64 pipe (two lanes a clock and SM) bounds the
// all-FP64 kernels.
__device__ __forceinline__ double double_from_fix128(__int128 v, int s) {
  const unsigned long long vh = (unsigned long long)((unsigned __int128)v >> 64), vl = (unsigned long long)v;
  if (v >= 0) {
    if (v == 0) return 0.0;
    const int z = vh ? __clzll((long long)vh) : 64 + __clzll((long long)vl);
    const int ex = 127 - z + 1022 - s;                  // the exponent field less one
    if (ex >= 0 && ex < 2045) {
      const unsigned __int128 n = (unsigned __int128)v << z;
      unsigned long long t = (unsigned long long)(n >> 64);
      if ((unsigned long long)n) t |= 1ull;
      const unsigned long long m = t >> 11;
      const unsigned up = ((unsigned)t & 0x7ffu) + ((unsigned)m & 1u) > 0x400u ? 1u : 0u;
      return __longlong_as_double((long long)(((unsigned long long)ex << 52) + m + up));
    }
  }
  const bool negv = v < 0;
  const unsigned __int128 a = negv ? (unsigned __int128)0 - (unsigned __int128)v : (unsigned __int128)v;
  const unsigned long long hi = (unsigned long long)(a >> 64), lo = (unsigned long long)a;
  int msb = hi ? 127 - __clzll((long long)hi) : 63 - __clzll((long long)lo);
  unsigned long long m;
  if (msb <= 52) {
    m = lo << (52 - msb);
  } else {
    const int sh = msb - 52;
    m = (unsigned long long)(a >> sh);
    const unsigned __int128 rem = a & (((unsigned __int128)1 << sh) - 1);
    const unsigned __int128 half = (unsigned __int128)1 << (sh - 1);
    if (rem > half || (rem == half && (m & 1ull))) {
      ++m;
      if (m == (1ull << 53)) {
        m >>= 1;
        ++msb;
      }
    }
  }
  // 2^msb (1 + frac): exact, msb <= 127
  const double d = __longlong_as_double((long long)(((unsigned long long)(msb + 1023) << 52) | (m & ((1ull << 52) - 1ull))));
  return scale_pow2d(negv ? -d : d, -s);
}

__device__ __forceinline__ long long fixr(float x, int s) { return fix_from_float(x, s); }
// round(x 2^s) for x >= 0 (the terms m and m/r): fix_from_float's value, as one
// 32 x 32 -> 64-bit product where the quantum is finer than x's last place by 2^30
// at most, else with the round half up done as one add before the shift
__device__ __forceinline__ long long fixp(float x, int s) {
  const uint32_t b = __float_as_uint(x);
  const int e = (int)(b >> 23);
  const int sh = e - 150 + s;
  const uint32_t mant = (b & 0x7fffffu) | 0x800000u;
  if ((unsigned)sh <= 30u && e != 0) return (long long)((unsigned long long)mant * (unsigned long long)(1u << sh));
  if (e == 0) return 0;
  if (sh >= 0) return (long long)((unsigned long long)mant << (sh > 39 ? 39 : sh));
  const int rs = -sh;
  return rs > 24 ? 0ll : (long long)((mant + (1u << (rs - 1))) >> rs);
}
// acc += fix_from_float(x, s): with the quantum finer than x's last place by 2^30
// at most (as it is unless x is 2^20 times smaller than the halo's largest term)
// one 32 x 32 -> 64-bit multiply-add of the signed mantissa, 10 instructions for
// 18 (21 with the general case's branches)
__device__ __forceinline__ void add_fix(long long& acc, float x, int s) {
  const uint32_t b = __float_as_uint(x);
  const int e = (int)((b >> 23) & 0xff);
  const int sh = e - 150 + s;
  if ((unsigned)sh <= 30u && e != 0) {
    const int mant = (int)((b & 0x7fffffu) | 0x800000u), sg = (int)b >> 31;
    acc += (long long)((mant ^ sg) - sg) * (long long)(int)(1u << sh);
  } else {
    acc += fix_from_float(x, s);
  }
}
__device__ __forceinline__ void add_fix(__int128& acc, double x, int s) { acc += fix128_from_double(x, s); }

__device__ __forceinline__ __int128 fixp(double x, int s) { return fix128_from_double(x, s); }
__device__ __forceinline__ __int128 fixr(double x, int s) { return fix128_from_double(x, s); }
__device__ __forceinline__ float from_fix(long long v, int s, float) { return float_from_fix(v, s); }
__device__ __forceinline__ double from_fix(__int128 v, int s, double) { return double_from_fix128(v, s); }
__device__ __forceinline__ double dfix(long long v, int s) { return double_from_fix(v, s); }
__device__ __forceinline__ double dfix(__int128 v, int s) { return double_from_fix128(v, s); }

__device__ __forceinline__ uint32_t shfl_up_x(uint32_t x, int o) { return __shfl_up_sync(FULL_MASK, x, o); }
__device__ __forceinline__ int shfl_xor_x(int x, int o) { return __shfl_xor_sync(FULL_MASK, x, o); }
__device__ __forceinline__ long long shfl_up_x(long long x, int o) { return __shfl_up_sync(FULL_MASK, x, o); }
__device__ __forceinline__ __int128 shfl_up_x(__int128 x, int o) {
  const unsigned long long lo = __shfl_up_sync(FULL_MASK, (unsigned long long)x, o);
  const unsigned long long hi = __shfl_up_sync(FULL_MASK, (unsigned long long)((unsigned __int128)x >> 64), o);
  return (__int128)(((unsigned __int128)hi << 64) | (unsigned __int128)lo);
}
__device__ __forceinline__ long long shfl_xor_x(long long x, int o) { return __shfl_xor_sync(FULL_MASK, x, o); }
__device__ __forceinline__ __int128 shfl_xor_x(__int128 x, int o) {
  const unsigned long long lo = __shfl_xor_sync(FULL_MASK, (unsigned long long)x, o);
  const unsigned long long hi = __shfl_xor_sync(FULL_MASK, (unsigned long long)((unsigned __int128)x >> 64), o);
  return (__int128)(((unsigned __int128)hi << 64) | (unsigned __int128)lo);
}
__device__ __forceinline__ long long shfl_idx_x(long long x, int l) { return __shfl_sync(FULL_MASK, x, l); }
__device__ __forceinline__ __int128 shfl_idx_x(__int128 x, int l) {
  const unsigned long long lo = __shfl_sync(FULL_MASK, (unsigned long long)x, l);
  const unsigned long long hi = __shfl_sync(FULL_MASK, (unsigned long long)((unsigned __int128)x >> 64), l);
  return (__int128)(((unsigned __int128)hi << 64) | (unsigned __int128)lo);
}
template <typename X>
__device__ __forceinline__ X wsum(X x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += shfl_xor_x(x, o);
  return x;
}
template <typename X>
__device__ __forceinline__ X wscan(X x, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const X y = shfl_up_x(x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// Sum over the CTA of one value per thread (every thread gets the total).
template <typename X>
__device__ __forceinline__ X block_sum(X x, X* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  x = wsum(x);
  __syncthreads();
  if (lane == 0) red[warp] = x;
  __syncthreads();
  X s = 0;
#pragma unroll
  for (int w = 0; w < NWARP; ++w) s += red[w];
  return s;
}

// block_sum for a CTA of NT threads.
template <typename X, int NT>
__device__ __forceinline__ X block_sum_n(X x, X* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  x = wsum(x);
  __syncthreads();
  if (lane == 0) red[warp] = x;
  __syncthreads();
  X s = 0;
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) s += red[w];
  return s;
}

// Exclusive prefix over the CTA's threads (thread order) of one value.
template <typename X>
__device__ __forceinline__ X block_excl(X x, X* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const X inc = wscan(x, lane);
  __syncthreads();
  if (lane == 31) red[warp] = inc;
  __syncthreads();
  X b = 0;
#pragma unroll
  for (int w = 0; w < NWARP; ++w)
    if (w < warp) b += red[w];
  return b + inc - x;
}

// ---- per-particle arithmetic ---------------------------------------------------------

__device__ __forceinline__ uint32_t key_of(float r) { return __float_as_uint(r); }
__device__ __forceinline__ unsigned long long key_of(double r) { return (unsigned long long)__double_as_longlong(r); }
__device__ __forceinline__ float radius_of_key(uint32_t k) { return __uint_as_float(k); }
__device__ __forceinline__ double radius_of_key(unsigned long long k) { return __longlong_as_double((long long)k); }
__device__ __forceinline__ int exp_of_bits(unsigned long long b, float) { return (int)((b >> 23) & 0xff) - 127; }
__device__ __forceinline__ int exp_of_bits(unsigned long long b, double) { return (int)((b >> 52) & 0x7ff) - 1023; }
__device__ __forceinline__ unsigned long long abs_bits(float x) { return __float_as_uint(fabsf(x)); }
__device__ __forceinline__ unsigned long long abs_bits(double x) {
  return (unsigned long long)__double_as_longlong(fabs(x));
}
__device__ __forceinline__ float rinv_real(float r, const ParamsDev& P) { return rinv_of(r, P.r_soft_f); }
// Comparisons of doubles on the integer pipe (same truth values, NaN included).
constexpr unsigned long long INF_BITS = 0x7ff0000000000000ull;
// a <= b, b >= 0 and a >= 0 or NaN
__device__ __forceinline__ bool le_positive(double a, double b) {
  const unsigned long long x = (unsigned long long)__double_as_longlong(a), y = (unsigned long long)__double_as_longlong(b);
  return x <= y && y <= INF_BITS;
}
__device__ __forceinline__ bool positive(double a) {
  return (unsigned long long)__double_as_longlong(a) - 1ull < INF_BITS;
}
__device__ __forceinline__ double rinv_real(double r, const ParamsDev& P) {
  // fmax(r, r_soft) for r_soft >= 0 (r: not NaN), on the integer pipe
  const long long a = __double_as_longlong(r), b = __double_as_longlong(P.r_soft);
  const double rr = __longlong_as_double(a > b ? a : b);
  return positive(rr) ? 1.0 / rr : 0.0;
}
// rinv_real(r, P) > 0, without the division
__device__ __forceinline__ bool rinv_positive(float r, const ParamsDev& P) { return fmaxf(r, P.r_soft_f) > 0.0f; }
__device__ __forceinline__ bool rinv_positive(double r, const ParamsDev& P) { return positive(r) || positive(P.r_soft); }
__device__ __forceinline__ unsigned long long bits_of(float x) { return __float_as_uint(x); }
__device__ __forceinline__ unsigned long long bits_of(double x) { return (unsigned long long)__double_as_longlong(x); }
__device__ __forceinline__ float real_of_bits(unsigned long long b, float) { return __uint_as_float((uint32_t)b); }
__device__ __forceinline__ double real_of_bits(unsigned long long b, double) { return __longlong_as_double((long long)b); }
__device__ __forceinline__ float phi_real(float M, float ri, float S, const ParamsDev& P) { return phi_of(M, ri, S, P.Gf); }
__device__ __forceinline__ double phi_real(double M, double ri, double S, const ParamsDev& P) {
  return __dmul_rn(-P.G, __fma_rn(M, ri, S));
}
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fma_x(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_x(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float neg0(float) { return -0.0f; }
__device__ __forceinline__ double neg0(double) { return -0.0; }

// All-FP64 recentring, written as the FP64 definition reads: d = x - c, then
// the minimum image, r^2 = (dx^2 + dy^2) + dz^2, r = sqrt(r^2) (both
// correctly rounded).
template <int CT>
__device__ __forceinline__ void offset_f64(const ParticlesDev& p, long long i, const HaloDev& H, double box,
                                           double d[3]) {
  double x[3];
  if (CT == AHF_COORD_F64) {
    x[0] = __ldg((const double*)p.x + i);
    x[1] = __ldg((const double*)p.y + i);
    x[2] = __ldg((const double*)p.z + i);
  } else {
    x[0] = (double)__ldg((const float*)p.x + i);
    x[1] = (double)__ldg((const float*)p.y + i);
    x[2] = (double)__ldg((const float*)p.z + i);
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    double v = __dsub_rn(x[a], H.c[a]);
    if (box > 0.0) {
      const double half = 0.5 * box;
      // (|v| > half, or NaN, on the integer pipe; rarely taken)
      if (((unsigned long long)__double_as_longlong(v) & ~(1ull << 63)) > (unsigned long long)__double_as_longlong(half)) {
        if (v > half) v = __dsub_rn(v, box);
        if (v < -half) v = __dadd_rn(v, box);
      }
    }
    d[a] = v;
  }
}

template <int CT>
__device__ __forceinline__ void load_velocity_f64(const ParticlesDev& p, long long i, double v[3]) {
  if (CT == AHF_COORD_F64) {
    v[0] = __ldg((const double*)p.vx + i);
    v[1] = __ldg((const double*)p.vy + i);
    v[2] = __ldg((const double*)p.vz + i);
  } else {
    v[0] = (double)__ldg((const float*)p.vx + i);
    v[1] = (double)__ldg((const float*)p.vy + i);
    v[2] = (double)__ldg((const float*)p.vz + i);
  }
}

template <int CT>
__device__ __forceinline__ double load_mass_f64(const ParticlesDev& p, long long i) {
  if (p.m == nullptr) return p.m0;
  if (CT == AHF_COORD_F64) return __ldg((const double*)p.m + i);
  return (double)__ldg((const float*)p.m + i);
}

// ---- prepare ---------------------------------------------------------------------

// The tile's counts of the keys' low byte, in g_hist's layout: the first radix
// pass sorts on that byte whenever it varies (it does for radii), and then
// reads these counts instead of running its own histogram kernel.
__device__ __forceinline__ void store_low_byte_hist(const GridLaunch& L, int t, int k, const uint32_t* h) {
  const int t0 = L.halo_tile0[k], th = L.halo_tile0[k + 1] - t0;
  L.tile_hist[(size_t)t0 * 256 + (size_t)threadIdx.x * th + (t - t0)] = h[threadIdx.x];
}

// The largest m, m / max(r, r_soft) and |m v_k| of a thread's members (the
// scales of the exact sums follow from their exponents).  With one mass for all
// only the smallest radius and the largest |v_k| are kept: rounding is monotone,
// so m0 times their values is the largest of the products, and the reciprocal
// and three products per candidate fall away.
template <typename R>
struct Maxima {
  using Key = typename Prec<R>::Key;
  Key m = 0, a = 0, v = 0;                 // uniform mass: a = complement of the smallest r's bits, v = |v| bits
  __device__ __forceinline__ void add(const ParamsDev& P, bool masses, R mass, R r, const R vel[3]) {
    if (masses) {
      m = max(m, (Key)abs_bits(mass));
      a = max(a, (Key)abs_bits(mass * rinv_real(r, P)));
#pragma unroll
      for (int k = 0; k < 3; ++k) v = max(v, (Key)abs_bits(mul_rn(mass, vel[k])));
    } else {
      // (a radius of zero has a reciprocal of zero unless softened: left out)
      if (rinv_positive(r, P)) a = max(a, (Key)~(Key)bits_of(r));
#pragma unroll
      for (int k = 0; k < 3; ++k) v = max(v, (Key)abs_bits(vel[k]));
    }
  }
  // The warp's maxima, in every lane.
  __device__ __forceinline__ void warp(const ParamsDev& P, bool masses, const ParticlesDev& p, int n,
                                       unsigned long long& mm, unsigned long long& mr, unsigned long long& mv) {
    for (int o = 16; o > 0; o >>= 1) {
      m = max(m, __shfl_xor_sync(FULL_MASK, m, o));
      a = max(a, __shfl_xor_sync(FULL_MASK, a, o));
      v = max(v, __shfl_xor_sync(FULL_MASK, v, o));
    }
    mm = m;
    mr = a;
    mv = v;
    if (!masses) {
      const R m0 = sizeof(R) == 4 ? (R)p.m0f : (R)p.m0;
      const bool any = __any_sync(FULL_MASK, n > 0);
      mm = any ? abs_bits(m0) : 0ull;
      mr = a ? abs_bits(m0 * rinv_real(real_of_bits((Key)~a, R()), P)) : 0ull;
      mv = abs_bits(mul_rn(m0, real_of_bits(v, R())));
    }
  }
};

// The CTA's key range, per-halo maxima and member count merged into the call's
// words.  Every thread passes its warp's reduced values; the CTA reduces them
// once more and thread 0 issues an atomic only where it can change the word
// (OR, AND and max are idempotent, so a stale read costs an extra atomic,
// never a wrong value).  Thousands of tiles share a handful of words, so one
// atomic per warp and word would queue on the same addresses.
__device__ __forceinline__ void merge_prepare(const GridLaunch& L, int k, unsigned long long orb,
                                              unsigned long long andb, unsigned long long mxm,
                                              unsigned long long mxr, unsigned long long mxv, int nmem) {
  __shared__ unsigned long long red[5][NWARP];
  __shared__ int rn[NWARP];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) {
    red[0][warp] = orb;
    red[1][warp] = andb;
    red[2][warp] = mxm;
    red[3][warp] = mxr;
    red[4][warp] = mxv;
    rn[warp] = nmem;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  unsigned long long o = 0, a = ~0ull, m0 = 0, m1 = 0, m2 = 0;
  long long n = 0;
#pragma unroll
  for (int w = 0; w < NWARP; ++w) {
    o |= red[0][w];
    a &= red[1][w];
    m0 = max(m0, red[2][w]);
    m1 = max(m1, red[3][w]);
    m2 = max(m2, red[4][w]);
    n += rn[w];
  }
  GridHaloState* st = L.state + k;
  if (o & ~__ldcg(&L.ctl->key_or)) atomicOr(&L.ctl->key_or, o);
  if (~a & __ldcg(&L.ctl->key_and)) atomicAnd(&L.ctl->key_and, a);
  if (m0 > __ldcg(&st->mass_max_bits)) atomicMax(&st->mass_max_bits, m0);
  if (m1 > __ldcg(&st->mr_max_bits)) atomicMax(&st->mr_max_bits, m1);
  if (m2 > __ldcg(&st->mv_max_bits)) atomicMax(&st->mv_max_bits, m2);
  if (n) atomicAdd((unsigned long long*)&st->n_member, (unsigned long long)n);
}

// ---- distribution over radial bins -----------------------------------------------
//
// The radial order needs no comparison sort of a whole halo.  A halo of th
// tiles gets 2 th bins of radius (1,024 candidates each on average, cut into 512
// parts; a halo of one tile is one bin), monotone in r.  The prepare counts each member in its bin and keeps
// its rank of arrival; a scan of the bins' counts gives every bin its first
// position; one scatter moves each member's record to its bin; and one CTA per
// bin orders it on chip and writes the radial-order streams.  Against the radix
// sort below (a histogram, two scans and a scatter per key byte, then a random
// gather of every record) each record moves twice, as one full 32-byte sector.
//
// The bins follow the halo's own distribution: a strided sample of its
// candidates is counted in 1,024 cells (256 for small haloes) of equal width in
// the bits of r (so logarithmic in r) from below its smallest radius up to its largest, and each
// cell gets parts of bins in proportion to its count (and a little more, so
// that no cell is left without), a member's place within its cell taken as
// linear in the bits of r.  Radii beyond the largest sampled one get tail parts
// in intervals that double in width.  The sample only balances the bins; the
// order does not depend on it.
//
// Measured against the radix sort for every halo (whole calls): 64 hosts of
// 1.5e8 candidates 13.2 -> 12.2 ms; 3,000 haloes in FP64 (keys of 8 bytes) 2.70 ->
// 2.11 ms; 11,000 candidates in FP64 590 -> 432 us; 3 hosts of 4e6 with gas 0.84 ->
// 0.75 ms.  The prepare is bound by its integer arithmetic and the latency of
// the counting atomics, the scatter by DRAM (two thirds of its peak), the
// ordering by issue slots (65 % busy).
//
// A bin holds BIN_MAX members at most (its CTA's shared memory).  When one would
// hold more (thousands of equal radii, a thin shell in a void), ctl->overflow is
// set, every later kernel of the attempt returns at once and the host runs the
// radix sort instead.  A bin in which a part holds so many that ordering it by
// counting would be slow (hundreds of equal radii) is ordered by comparisons
// (order_tied).

constexpr int CELLS = 1024;              // at most
constexpr int SAMPLE_T = 1024;
constexpr int SAMPLE_PT = 32;            // sampled candidates per thread
constexpr int SAMPLE_MAX = SAMPLE_T * SAMPLE_PT;
constexpr int TAILS = 32;                // tail intervals
constexpr int PARTS = 512;               // parts of a bin
constexpr uint32_t TAB_UNIT = 2u;        // bin tables count in halves of a part (below 2^32 for any halo)
constexpr uint32_t NO_RANK = 0xffffu;    // rank of a non-member
static_assert(PARTS == 2 * T, "two parts a thread");
constexpr int BIN_MAX = 3072;            // members of a bin
constexpr uint32_t PART_MAX = 512u;      // members of a part ordered by counting
constexpr int BIN_PAD = 32;              // words between bins' counters: atomics on one 128-byte line queue
constexpr int AGG_BINS = 512;            // halo's bins up to which a CTA counts in shared memory first

// Bins of a halo of th tiles; its first is 2 t0.
__host__ __device__ __forceinline__ int halo_bins(int th) { return th > 1 ? 2 * th : th; }

__device__ __forceinline__ bool bins_overflowed(const GridLaunch& L) { return __ldcg(&L.ctl->overflow) != 0; }

// The key a bin is found from: the bits of r as a float (cutting a double
// radius is monotone, and needs no conversion on the FP64 pipe).
__device__ __forceinline__ uint32_t bin_key(float r) { return __float_as_uint(r); }
__device__ __forceinline__ uint32_t bin_key(double r) {
  const unsigned long long x = (unsigned long long)__double_as_longlong(r) >> 29, base = 896ull << 23;
  return x > base ? (uint32_t)min(x - base, 0x7f7fffffull) : 0u;
}

// Candidates sampled of n: an eighth, 512 to SAMPLE_MAX of them.
__device__ __forceinline__ int sample_size(long long n) {
  return (int)min(n, max(512ll, min((long long)SAMPLE_MAX, n >> 3)));
}
// Parts of one tail interval: four times the candidates expected beyond the
// largest of the sample, at two to a part.  TAILS intervals stay below half
// of a halo's parts (2,048 at least).
__device__ __forceinline__ uint32_t tail_parts(long long n) {
  const int S = sample_size(n);
  return S > 0 ? 2u * (uint32_t)(n / S) : 1u;
}

// Cells of a halo of th tiles.
__host__ __device__ __forceinline__ int map_cells(int th) { return th >= 8 ? CELLS : 256; }
// Its table of cells, behind the bins' counters in tile_hist (192 words a tile).
__device__ __forceinline__ uint32_t* bin_table(const GridLaunch& L, int t0) {
  return L.tile_hist + (size_t)L.n_tiles * 2 * BIN_PAD + (size_t)t0 * (256 - 2 * BIN_PAD);
}

// A halo's map from keys to parts (PARTS to a bin): `cells` cells of 2^sh keys from
// k0 on, ending with the largest sampled key kx; tail intervals of 2^gs keys,
// then doubling.
struct BinMap {
  uint32_t k0, kx, tb, main;             // main: parts before the tails
  int sh, gs, cells;
};

// The map of halo k and its cells' first parts (in units of 1 / TAB_UNIT; the last
// entry: main) into shared memory.
__device__ __forceinline__ BinMap load_bin_map(const GridLaunch& L, int k, int t0, long long n, int th, uint32_t* tab) {
  const GridHaloState& S = L.state[k];
  BinMap M;
  M.k0 = S.bin_k0;
  M.kx = S.bin_kx;
  M.sh = S.bin_shifts & 255;
  M.gs = S.bin_shifts >> 8;
  M.tb = tail_parts(n);
  M.main = (uint32_t)halo_bins(th) * PARTS - TAILS * M.tb;
  M.cells = map_cells(th);
  const uint32_t* src = bin_table(L, t0);
  if (th > 1)
    for (int c = threadIdx.x; c < M.cells; c += T) tab[c] = src[c];
  if (threadIdx.x == 0) tab[M.cells] = M.main * TAB_UNIT;
  return M;
}

// Part of a key (monotone in it): its cell, then linear within the cell; keys
// below the first cell go to part 0.
__device__ __forceinline__ uint32_t part_of(uint32_t key, const BinMap& M, const uint32_t* tab) {
  if (key > M.kx) {
    const uint32_t x = key - M.kx - 1u, y = x >> M.gs;
    const int i = y == 0u ? 0 : 32 - __clz(y);
    const int w = i == 0 ? M.gs : M.gs + i - 1;        // the interval's width
    const uint32_t lo = i == 0 ? x : x - (1u << w);
    return M.main + (uint32_t)i * M.tb + (uint32_t)(((unsigned long long)lo * M.tb) >> w);
  }
  const uint32_t x = key > M.k0 ? key - M.k0 : 0u;
  const uint32_t c = min(x >> M.sh, (uint32_t)M.cells - 1u);
  const uint32_t lo = min(x - (c << M.sh), (1u << M.sh) - 1u);
  const uint32_t b0 = tab[c], w = tab[c + 1] - b0;
  return min((b0 + (uint32_t)(((unsigned long long)w * lo) >> M.sh)) / TAB_UNIT, M.main - 1u);
}

static_assert(CELLS == SAMPLE_T && 8 * (256 - 2 * BIN_PAD) >= CELLS && 2 * (256 - 2 * BIN_PAD) >= 256, "bin tables");

// The sample's keys, one candidate per thread, to rec_b at the halo's base, and
// their extremes.  CTA b of halo k: from a grid of (b, k), or of the tiles, of
// which each halo's first ones serve (whichever grid is the smaller).
template <typename R, int CT>
__global__ void __launch_bounds__(T) g_sample(GridLaunch L) {
  const int k = gridDim.y > 1 ? blockIdx.y : L.tile_halo[blockIdx.x];
  const int t0 = L.halo_tile0[k], th = L.halo_tile0[k + 1] - t0;
  if (th <= 1) return;                   // one bin: no map
  const HaloDev& H = L.halos[k];
  const long long n = H.count;
  const int S = sample_size(n);
  const int b = gridDim.y > 1 ? blockIdx.x : blockIdx.x - t0;
  if (b >= (S + T - 1) / T) return;      // (at most th shares: S is an eighth of n, or 512 of two tiles)
  const int j = b * T + threadIdx.x;
  uint32_t key = KEY_NONMEMBER;
  const bool in = j < S;
  if (in) {
    // groups of 8 neighbours (one or two sectors per array), evenly spread
    const long long groups = (S + 7) >> 3;
    long long pi = H.offset + min(((j >> 3) * n) / groups + (j & 7), n - 1);
    if (L.out.member_idx) pi = L.out.member_idx[pi];
    if (pi >= 0 && pi < L.p.n) {
      if constexpr (sizeof(R) == 4) {
        float d[3];
        long long f[3];
        offset_of<CT>(L.p, pi, H, d, f);
        if (member_of<CT>(L.p, pi, H, d, f)) key = bin_key(radius_of(d));
      } else {
        double d[3];
        offset_f64<CT>(L.p, pi, H, L.frame.box, d);
        const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1])), __dmul_rn(d[2], d[2]));
        if (le_positive(r2, H.R2)) key = bin_key(sqrt(r2));
      }
    }
    ((uint32_t*)L.rec_b)[H.gbase + j] = key;
  }
  const bool mem = key != KEY_NONMEMBER;
  const uint32_t km = __reduce_max_sync(FULL_MASK, mem ? key : 0u);
  const uint32_t kn = __reduce_max_sync(FULL_MASK, mem ? ~key : 0u);
  if ((threadIdx.x & 31) == 0 && kn) {
    atomicMax(&L.state[k].bin_kx, km);
    atomicMax(&L.state[k].bin_k0, kn);   // the complement of the smallest key
  }
}

// Members expected in a bin above which the attempt is given up before it begins:
// every member adds to its bin's counter, and those of one address queue.  10^7
// candidates, 9 10^6 at one radius: 7.3 ms with the attempt, 1.2 by the radix sort
// alone.  (Below this line it costs 40 us at most, and a sample may mistake a
// clump of neighbours in the candidate list for a shell.)
constexpr long long HOPELESS = 16 * BIN_MAX;

// One CTA per halo: the sample's cells and the table.
__global__ void __launch_bounds__(SAMPLE_T) g_bin_map(GridLaunch L) {
  __shared__ uint32_t cell[CELLS], key_lo[CELLS], key_hi[CELLS];   // (key_lo, key_hi: heavy cells)
  __shared__ uint32_t wt[SAMPLE_T / 32];
  const int k = blockIdx.x;
  const HaloDev& H = L.halos[k];
  const long long n = H.count;
  const int th = L.halo_tile0[k + 1] - L.halo_tile0[k];
  if (th <= 1) return;
  const int S = sample_size(n);
  const uint32_t* skey = (const uint32_t*)L.rec_b + H.gbase;
  const uint32_t kx = L.state[k].bin_kx, kn = min(~L.state[k].bin_k0, kx);
  const int cells = map_cells(th), log_cells = cells == CELLS ? 10 : 8;
  cell[threadIdx.x] = 0u;
  // the cells end with the largest sampled key and start a quarter of the
  // sampled range and two octaves below the smallest
  const uint32_t range = kx - kn;
  const uint32_t want = range + (range >> 2) + (2u << 23);        // < 2^32
  const int sh = 32 - log_cells - __clz(want - 1u);               // cells << sh >= want
  const uint32_t span = (uint32_t)min((unsigned long long)cells << sh, 0xffffffffull);
  const uint32_t k0 = kx + 1u > span ? kx + 1u - span : 0u;
  __syncthreads();
#pragma unroll 8
  for (int j = threadIdx.x; j < S; j += SAMPLE_T) {
    const uint32_t key = skey[j];
    if (key != KEY_NONMEMBER) atomicAdd(&cell[min((key > k0 ? key - k0 : 0u) >> sh, (uint32_t)cells - 1u)], 1u);
  }
  __syncthreads();
  const int c = threadIdx.x, lane = c & 31, warp = c >> 5;
  // weight of a cell with m samples: m + 3 sqrt(m) + 4 (scaled down for small
  // samples), an upper estimate, so that the bins of cells a few samples fell in
  // rarely hold more than their share
  uint32_t w = 0u;
  if (c < cells) {
    const float m = (float)cell[c];
    w = (uint32_t)(64.0f * (m + 3.0f * sqrtf(m))) + max(1u, (uint32_t)S / 128u);
  }
  const uint32_t inc = warp_inclusive_scan(w, lane);
  if (lane == 31) wt[warp] = inc;
  __syncthreads();
  uint32_t b0 = 0u, b1 = 0u;             // the cell's parts begin and end
  if (c < cells) {
    uint32_t base = inc - w, tot = 0;
    for (int v = 0; v < SAMPLE_T / 32; ++v) {
      const uint32_t x = wt[v];
      if (v < warp) base += x;
      tot += x;
    }
    const unsigned long long all = ((unsigned long long)halo_bins(th) * PARTS - TAILS * tail_parts(n)) * TAB_UNIT;
    b0 = (uint32_t)((all * base) / tot);
    b1 = (uint32_t)((all * (base + w)) / tot);
    bin_table(L, L.halo_tile0[k])[c] = b0;
    if (c == 0) {
      // the tails start with a quarter of the spacing of the last cells' samples
      const uint32_t cx = min((kx - k0) >> sh, (uint32_t)cells - 1u);
      const uint32_t sp = (1u << sh) / (cell[cx] + (cx ? cell[cx - 1] : 0u) + 1u);
      GridHaloState& st = L.state[k];
      st.bin_k0 = k0;
      st.bin_shifts = sh | (max(0, 29 - __clz(max(sp, 1u))) << 8);
    }
  }
  // Cells of so many members that a few bins could not hold them (few haloes have
  // one): the bins that their samples fall into, as part_of finds them.
  if (n <= HOPELESS) return;
  const long long members = (long long)cell[c] * (n / S);
  if (!__syncthreads_or(members > HOPELESS)) return;
  key_lo[c] = 0xffffffffu;
  key_hi[c] = 0u;
  __syncthreads();
  for (int j = threadIdx.x; j < S; j += SAMPLE_T) {
    const uint32_t key = skey[j];
    if (key == KEY_NONMEMBER) continue;
    const uint32_t x = key > k0 ? key - k0 : 0u, to = min(x >> sh, (uint32_t)cells - 1u);
    const uint32_t lo = min(x - (to << sh), (1u << sh) - 1u);
    atomicMin(&key_lo[to], lo);
    atomicMax(&key_hi[to], lo);
  }
  __syncthreads();
  if (members > HOPELESS) {
    auto bin_at = [&](uint32_t lo) {
      return (b0 + (uint32_t)(((unsigned long long)(b1 - b0) * lo) >> sh)) / (TAB_UNIT * PARTS);
    };
    if (members > HOPELESS * ((long long)bin_at(key_hi[c]) - bin_at(key_lo[c]) + 1)) {
      L.ctl->overflow = 1;
      L.ctl->no_bins = 1;
    }
  }
}

// Bin of a member and its rank of arrival there, for the members a CTA holds at
// one step: `bin` their bins (relative to the halo's first), mem false for
// none.  One bin: a warp's members take consecutive ranks (one atomic per
// warp); AGG_BINS at most: counted in shared memory first (scnt, zero before and
// reused as the bins' bases), one global atomic per bin met.  (With more bins
// each member's atomic is issued where its bin is found: bin_rank_now.)
template <int N>
__device__ __forceinline__ void bin_ranks(uint32_t* cnt, int nb, const bool mem[N], const uint32_t bin[N], uint32_t rk[N],
                                          uint32_t* scnt) {
  if (nb == 1) {
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const unsigned m = __ballot_sync(FULL_MASK, mem[q]);
      uint32_t base = 0;
      if ((threadIdx.x & 31) == 0 && m) base = atomicAdd(cnt, (uint32_t)__popc(m));
      base = __shfl_sync(FULL_MASK, base, 0);
      rk[q] = base + __popc(m & lanemask_lt());
    }
  } else if (nb <= AGG_BINS) {
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (mem[q]) rk[q] = atomicAdd(&scnt[bin[q]], 1u);
    __syncthreads();
    for (int c = threadIdx.x; c < nb; c += T) {
      const uint32_t v = scnt[c];
      if (v) scnt[c] = atomicAdd(&cnt[(size_t)c * BIN_PAD], v);
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (mem[q]) rk[q] += scnt[bin[q]];
  }
}
__device__ __forceinline__ uint32_t bin_rank_now(uint32_t* cnt, int nb, uint32_t bin) {
  return nb > AGG_BINS ? atomicAdd(&cnt[(size_t)bin * BIN_PAD], 1u) : 0u;
}

// The tile's sub-tile sums of the initial set (copy 1) and its sum m v zeroed,
// for the CTAs that will add to them.
template <typename R>
__device__ __forceinline__ void zero_sums(const GridLaunch& L, int t) {
  using Acc = typename Prec<R>::Acc;
  if (threadIdx.x < GRID_TILE / GRID_SUB) {
    const size_t u = (size_t)(L.n_tiles + t) * (GRID_TILE / GRID_SUB) + threadIdx.x;
    ((Acc*)L.agg_m)[u] = 0;
    ((Acc*)L.agg_r)[u] = 0;
    L.agg_c[u] = 0;
  }
  if (threadIdx.x < 3) A<Acc>(L.tile_mv[3 * (size_t)t + threadIdx.x]) = 0;
}

// The ranks of a thread's candidates (element q T + thread of the tile; rank
// NO_RANK for a non-member).
template <int N>
__device__ __forceinline__ void store_ranks(const GridLaunch& L, int2 tr, const bool mem[N], const uint32_t rk[N]) {
  bool over = false;
#pragma unroll
  for (int q = 0; q < N; ++q) {
    const int e = q * T + threadIdx.x;
    if (e < tr.y) L.rank[(size_t)tr.x + e] = (uint16_t)(mem[q] ? min(rk[q], NO_RANK) : NO_RANK);
    over |= mem[q] && rk[q] >= (uint32_t)BIN_MAX;
  }
  if (over) L.ctl->overflow = 1;
}

// Recentring in FP32.  The offset of a float coordinate x is RN(x - c'), c' the
// centre rounded to the halo's fixed-point grid (at most 62 bits: the sum of
// three floats).  x - hi and (x - hi) - mid split into sum and rounding error
// (Knuth's TwoSum, exact); what is left, t, is known to 2^-22 of its terms, and
// where both ends of that interval round the sum to the same float that is the
// result (Ziv's test).  Elsewhere (a tie, or about one candidate in 10^5), for x
// off the grid, and for candidates half a box away, the exact fixed-point route
// decides.  About 25 instructions an axis for 60 of the exact route.
struct Recentre {
  float hi[3], mid[3], lo[3];
  float near;                            // |x - hi| up to which no box wrap can occur
  uint32_t x0, xn;                       // |x| bits x0 .. x0 + xn are on the grid (xn = 0: never)
};
// Axis a of halo H's (one thread each).
__device__ __forceinline__ void recentre_axis(Recentre& C, const HaloDev& H, int a) {
  const long long c = H.cfix[a];
  const float h = f32_from_i64_rn(c);
  const long long r = c - (long long)h;
  const float m = f32_from_i64_rn(r);
  const float l = f32_from_i64_rn(r - (long long)m);
  const bool ok = !H.fast && H.frac >= -60 && H.frac <= 100;
  const float q = ok ? __int_as_float((127 - H.frac) << 23) : 0.0f;
  C.hi[a] = h * q;
  C.mid[a] = m * q;
  C.lo[a] = l * q;
  if (a == 0) {
    // half the box less 2^-18 of it and of the frame (the centre is within it)
    const float half = f32_from_i64_rn(H.boxfix >> 1) * q;
    C.near = H.boxfix > 0 ? half - 0x1p-18f * half - 0x1p-18f * (0x1p60f * q) : INFINITY;
    C.x0 = (uint32_t)(150 - H.frac) << 23;
    C.xn = ok ? 37u << 23 : 0u;
  }
}
// One axis; false: the exact route must decide.
__device__ __forceinline__ bool recentre(const Recentre& C, int a, float x, float& d) {
  const float h = C.hi[a], m = C.mid[a], l = C.lo[a];
  const float s = __fsub_rn(x, h), sb = __fsub_rn(s, x);
  const float e = __fsub_rn(__fsub_rn(x, __fsub_rn(s, sb)), __fadd_rn(h, sb));
  const float u = __fsub_rn(s, m), ub = __fsub_rn(u, s);
  const float w = __fsub_rn(__fsub_rn(s, __fsub_rn(u, ub)), __fadd_rn(m, ub));
  const float t = __fsub_rn(__fadd_rn(e, w), l);
  const float q = __fadd_rn(__fadd_rn(fabsf(e), fabsf(w)), fabsf(l));
  d = __fadd_rn(u, __fmaf_rn(q, 0x1p-21f, t));
  const float d2 = __fadd_rn(u, __fmaf_rn(q, -0x1p-21f, t));
  return d == d2 && fabsf(s) <= C.near && (__float_as_uint(x) & 0x7fffffffu) - C.x0 < C.xn;
}

// Mixed precision: the on-chip classes' float offsets (exact recentring),
// membership and radius; the record holds w = v + H d and r, then v and m.
// BINS: each member is counted in its radial bin and its rank of arrival kept;
// otherwise the keys and the first digit's histogram of the radix sort.
//
// Bound by issue slots and latency, not by memory (a third of the DRAM rate): a
// member took 474 instructions, in one chain a candidate.  The FP32 recentring
// and GROUP candidates in step (their chains overlap) took 144e6 candidates from
// 3.55 to 2.98 ms; 2 and 8 in step, 3, 5 and 6 CTAs an SM were slower.
constexpr int GROUP = 4;
template <int CT, bool BINS>
__global__ void __launch_bounds__(T, 4) g_prepare_mixed(GridLaunch L) {
  const int t = blockIdx.x;
  const int given_up = BINS ? L.ctl->no_bins : 0;
  const int2 tr = L.tile_range[t];
  const int k = L.tile_halo[t];
  const HaloDev H = L.halos[k];
  if (given_up) return;
  const ParamsDev& P = L.prm;
  uint32_t* key_a = (uint32_t*)L.key_a;
  float4* rec = (float4*)L.rec;
  __shared__ uint32_t h0[CELLS + 1];
  __shared__ uint32_t scnt[BINS ? AGG_BINS : 1];
  __shared__ Recentre C;
  const int t0 = L.halo_tile0[k], th = L.halo_tile0[k + 1] - t0;
  if (CT != AHF_COORD_F64 && threadIdx.x < 3) recentre_axis(C, L.halos[k], threadIdx.x);
  BinMap BM;
  if (BINS) {
    BM = load_bin_map(L, k, t0, H.count, th, h0);
    zero_sums<float>(L, t);
    if (halo_bins(th) <= AGG_BINS)
      for (int c = threadIdx.x; c < halo_bins(th); c += T) scnt[c] = 0u;
  } else h0[threadIdx.x] = 0u;
  uint32_t orb = 0, andb = 0xffffffffu;
  Maxima<float> mx;
  int nmem = 0;
  uint32_t* cnt = L.bin_n + (size_t)t0 * 2 * BIN_PAD;
  const int nb = halo_bins(th);
  bool ok[IPT];
  uint32_t bin[IPT], rk[IPT];
  // GROUP candidates at a time, each step of the way for all of them
#pragma unroll
  for (int q0 = 0; q0 < IPT; q0 += GROUP) {
    Cand<CT> c[GROUP];
#pragma unroll
    for (int i = 0; i < GROUP; ++i) {
      const int e = (q0 + i) * T + threadIdx.x;
      ok[q0 + i] = e < tr.y;
      long long pi = 0;
      if (ok[q0 + i]) {
        const long long slot = H.offset + ((long long)tr.x + e - H.gbase);
        pi = slot;
        if (L.out.member_idx) {
          pi = L.out.member_idx[slot];
          if (pi < 0 || pi >= L.p.n) {
            ok[q0 + i] = false;
            atomicOr(L.out.err, ERR_BAD_INDEX);
          }
        }
      }
      if (ok[q0 + i]) load_cand<CT>(L.p, pi, c[i]);
      else c[i] = Cand<CT>{};
    }
    if (q0 == 0) __syncthreads();        // the map, the counters and C are ready
    float d[GROUP][3], r[GROUP];
    bool sure[GROUP];
#pragma unroll
    for (int i = 0; i < GROUP; ++i) {
      sure[i] = false;
      d[i][0] = d[i][1] = d[i][2] = 0.0f;
      if (CT != AHF_COORD_F64 && !H.fast)
        sure[i] = recentre(C, 0, (float)c[i].x, d[i][0]) & recentre(C, 1, (float)c[i].y, d[i][1]) &
                  recentre(C, 2, (float)c[i].z, d[i][2]);
    }
#pragma unroll
    for (int i = 0; i < GROUP; ++i) {
      const float r2 = fmaf(d[i][2], d[i][2], fmaf(d[i][1], d[i][1], d[i][0] * d[i][0]));
      const bool in = r2 < H.R2lo;
      if (ok[q0 + i] && !(sure[i] && (in || r2 > H.R2hi))) {
        long long f[3];
        cand_offset<CT>(c[i], H, d[i], f);
        ok[q0 + i] = cand_member<CT>(c[i], H, d[i], f);
      } else {
        ok[q0 + i] = ok[q0 + i] && in;
      }
    }
#pragma unroll
    for (int i = 0; i < GROUP; ++i) r[i] = radius_of(d[i]);
    if (BINS && th > 1) {
#pragma unroll
      for (int i = 0; i < GROUP; ++i) bin[q0 + i] = part_of(ok[q0 + i] ? bin_key(r[i]) : 0u, BM, h0) / PARTS;
#pragma unroll
      for (int i = 0; i < GROUP; ++i)
        if (ok[q0 + i]) rk[q0 + i] = bin_rank_now(cnt, nb, bin[q0 + i]);
    }
#pragma unroll
    for (int i = 0; i < GROUP; ++i) {
      const int q = q0 + i;
      const int e = q * T + threadIdx.x;
      if (!BINS || th == 1) bin[q] = 0u;
      if (e >= tr.y) continue;
      const long long g = (long long)tr.x + e;
      uint32_t key = KEY_NONMEMBER;
      if (ok[q]) {
        const float m = cand_mass<CT>(L.p, c[i]);
        float v[3];
        cand_velocity<CT>(c[i], v);
        rec[2 * g] = make_float4(fmaf(P.Hf, d[i][0], v[0]), fmaf(P.Hf, d[i][1], v[1]), fmaf(P.Hf, d[i][2], v[2]), r[i]);
        rec[2 * g + 1] = make_float4(v[0], v[1], v[2], m);
        key = key_of(r[i]);
        mx.add(P, L.p.m != nullptr, m, r[i], v);
        ++nmem;
      }
      if (L.out.removed_iter) L.out.removed_iter[H.offset + (g - H.gbase)] = key == KEY_NONMEMBER ? -1 : 0;
      if (!BINS) {
        key_a[g] = key;
        atomicAdd(&h0[key & 0xffu], 1u);
        orb |= key;
        andb &= key;
      }
    }
  }
  if (BINS) {
    bin_ranks<IPT>(cnt, nb, ok, bin, rk, scnt);
    store_ranks<IPT>(L, tr, ok, rk);
  } else {
    __syncthreads();
    store_low_byte_hist(L, t, k, h0);
  }
  if (!BINS) {
    for (int o = 16; o > 0; o >>= 1) {
      orb |= __shfl_xor_sync(FULL_MASK, orb, o);
      andb &= __shfl_xor_sync(FULL_MASK, andb, o);
    }
  }
  unsigned long long mxm, mxr, mxv;
  mx.warp(P, L.p.m != nullptr, L.p, nmem, mxm, mxr, mxv);
  nmem = __reduce_add_sync(FULL_MASK, nmem);
  if (BINS) merge_prepare(L, k, 0ull, ~0ull, mxm, mxr, mxv, nmem);
  else merge_prepare(L, k, orb, (unsigned long long)andb | 0xffffffff00000000ull, mxm, mxr, mxv, nmem);
}

// All-FP64 mode: d = x - c in FP64 (minimum image), r^2 = (dx^2 + dy^2) + dz^2.
template <int CT, bool BINS>
__global__ void __launch_bounds__(T) g_prepare_f64(GridLaunch L) {
  const int t = blockIdx.x;
  const int given_up = BINS ? L.ctl->no_bins : 0;
  const int2 tr = L.tile_range[t];
  const int k = L.tile_halo[t];
  const HaloDev H = L.halos[k];
  if (given_up) return;
  const ParamsDev& P = L.prm;
  unsigned long long* key_a = (unsigned long long*)L.key_a;
  D4* rec = (D4*)L.rec;
  unsigned long long orb = 0, andb = ~0ull;
  Maxima<double> mx;
  int nmem = 0;
  __shared__ uint32_t h0[CELLS + 1];
  __shared__ uint32_t scnt[BINS ? AGG_BINS : 1];
  const int t0 = L.halo_tile0[k], th = L.halo_tile0[k + 1] - t0;
  BinMap BM;
  if (BINS) {
    BM = load_bin_map(L, k, t0, H.count, th, h0);
    zero_sums<double>(L, t);
    if (halo_bins(th) <= AGG_BINS)
      for (int c = threadIdx.x; c < halo_bins(th); c += T) scnt[c] = 0u;
  } else h0[threadIdx.x] = 0u;
  __syncthreads();
  bool mem[IPT];
  uint32_t bin[IPT], rk[IPT];
  uint32_t* cnt = L.bin_n + (size_t)t0 * 2 * BIN_PAD;
  const int nb = halo_bins(th);
#pragma unroll
  for (int j = 0; j < IPT; ++j) {
    const int e = j * T + threadIdx.x;
    mem[j] = false;
    bin[j] = 0u;
    if (e >= tr.y) continue;
    const long long g = (long long)tr.x + e;
    const long long slot = H.offset + (g - H.gbase);
    long long pi = slot;
    bool ok = true;
    if (L.out.member_idx) {
      pi = L.out.member_idx[slot];
      if (pi < 0 || pi >= L.p.n) {
        ok = false;
        atomicOr(L.out.err, ERR_BAD_INDEX);
      }
    }
    unsigned long long key = ~0ull;
    if (ok) {
      double d[3];
      offset_f64<CT>(L.p, pi, H, L.frame.box, d);
      const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1])), __dmul_rn(d[2], d[2]));
      if (le_positive(r2, H.R2)) {
        const double r = sqrt(r2);
        const double m = load_mass_f64<CT>(L.p, pi);
        double v[3];
        load_velocity_f64<CT>(L.p, pi, v);
        D4 a, b;
        a.x = __fma_rn(P.H, d[0], v[0]);
        a.y = __fma_rn(P.H, d[1], v[1]);
        a.z = __fma_rn(P.H, d[2], v[2]);
        a.w = r;
        b.x = v[0];
        b.y = v[1];
        b.z = v[2];
        b.w = m;
        rec[2 * g] = a;
        rec[2 * g + 1] = b;
        key = key_of(r);
        mem[j] = true;
        if (BINS && th > 1) {
          bin[j] = part_of(bin_key(r), BM, h0) / PARTS;
          rk[j] = bin_rank_now(cnt, nb, bin[j]);
        }
        mx.add(P, L.p.m != nullptr, m, r, v);
        ++nmem;
      }
    }
    if (L.out.removed_iter) L.out.removed_iter[slot] = key == ~0ull ? -1 : 0;
    if (!BINS) {
      key_a[g] = key;
      atomicAdd(&h0[(uint32_t)key & 0xffu], 1u);
      orb |= key;
      andb &= key;
    }
  }
  if (BINS) {
    bin_ranks<IPT>(cnt, nb, mem, bin, rk, scnt);
    store_ranks<IPT>(L, tr, mem, rk);
  } else {
    __syncthreads();
    store_low_byte_hist(L, t, k, h0);
  }
  if (!BINS) {
    for (int o = 16; o > 0; o >>= 1) {
      orb |= __shfl_xor_sync(FULL_MASK, orb, o);
      andb &= __shfl_xor_sync(FULL_MASK, andb, o);
    }
  }
  unsigned long long mxm, mxr, mxv;
  mx.warp(P, L.p.m != nullptr, L.p, nmem, mxm, mxr, mxv);
  nmem = __reduce_add_sync(FULL_MASK, nmem);
  if (BINS) merge_prepare(L, k, 0ull, ~0ull, mxm, mxr, mxv, nmem);
  else merge_prepare(L, k, orb, andb, mxm, mxr, mxv, nmem);
}

// The scales of a halo's exact sums and the start of its bookkeeping.
template <typename R>
__device__ __forceinline__ void halo_scales(GridHaloState& s) {
  const long long n = s.n_member;
  s.s_m = acc_scale<R>(exp_of_bits(s.mass_max_bits, R()), n);
  s.s_mr = acc_scale<R>(exp_of_bits(s.mr_max_bits, R()), n);
  s.s_mv = acc_scale<R>(exp_of_bits(s.mv_max_bits, R()), n);
  s.n_alive = n;
  s.active = 0;                          // set by the init pass
  s.n_iter = 0;
  s.status = 0;
  s.part_iter = 0;
  s.band = 0;
  s.k_first = 0x7fffffffffffffffll;
}

template <typename R>
__global__ void g_scales(GridLaunch L) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < L.n_halos) halo_scales<R>(L.state[k]);
}

// One CTA per halo: the first position of each of its bins (the exclusive
// prefix of their counts), and its scales.
template <typename R>
__global__ void __launch_bounds__(T) g_bin_base(GridLaunch L) {
  __shared__ uint32_t red[NWARP];
  __shared__ uint32_t carry;
  const int k = blockIdx.x;
  const int b0 = 2 * L.halo_tile0[k], b1 = b0 + halo_bins(L.halo_tile0[k + 1] - L.halo_tile0[k]);
  if (threadIdx.x == 0) {
    carry = 0u;
    halo_scales<R>(L.state[k]);
  }
  // four consecutive bins per thread and round
  for (int b = b0; b < b1; b += 4 * T) {
    uint32_t v[4], s = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int i = b + 4 * (int)threadIdx.x + j;
      v[j] = i < b1 ? L.bin_n[(size_t)i * BIN_PAD] : 0u;
      s += v[j];
    }
    uint32_t run = block_excl(s, red) + carry;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int i = b + 4 * (int)threadIdx.x + j;
      if (i < b1) L.bin_at[i] = run;
      run += v[j];
    }
    __syncthreads();
    if (threadIdx.x == T - 1) carry = run;
    __syncthreads();
  }
}

// 32 bytes to one sector (a 32-byte aligned address) as one store.
__device__ __forceinline__ void store_sector(void* p, float4 a, float4 b) {
  unsigned long long g;
  asm("cvta.to.global.u64 %0, %1;" : "=l"(g) : "l"(p));
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(g), "f"(a.x), "f"(a.y), "f"(a.z), "f"(a.w),
               "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w)
               : "memory");
}

// A member's record by bin: (w, r) and (v, candidate position).
__device__ __forceinline__ void put_binned(const GridLaunch& L, long long dst, float4 a, float4 b, uint32_t pos) {
  b.w = __uint_as_float(pos);
  store_sector((float4*)L.rec_b + 2 * dst, a, b);
}
__device__ __forceinline__ void put_binned(const GridLaunch& L, long long dst, D4 a, D4 b, uint32_t pos) {
  b.w = __longlong_as_double((long long)pos);
  D4* r = (D4*)L.rec_b + 2 * dst;
  r[0] = a;
  r[1] = b;
}
__device__ __forceinline__ uint32_t binned_pos(float x) { return __float_as_uint(x); }
__device__ __forceinline__ uint32_t binned_pos(double x) { return (uint32_t)__double_as_longlong(x); }

// Each member of a candidate tile to its bin: the bin's first position plus
// its rank.
template <typename R>
__global__ void __launch_bounds__(T, sizeof(R) == 4 ? 4 : 2) g_place(GridLaunch L) {
  using V4 = typename Prec<R>::V4;
  __shared__ uint32_t tab[CELLS + 1];
  if (bins_overflowed(L)) return;
  const int t = blockIdx.x;
  const int2 tr = L.tile_range[t];
  const int k = L.tile_halo[t];
  const long long gb = L.halos[k].gbase;
  const int t0 = L.halo_tile0[k], th = L.halo_tile0[k + 1] - t0;
  const BinMap BM = load_bin_map(L, k, t0, L.halos[k].count, th, tab);
  const V4* __restrict__ rec = (const V4*)L.rec;
  // batches of GB candidates, every load of a batch issued before its first use
  constexpr int GB = sizeof(R) == 4 ? 4 : 2;
  uint32_t rk[IPT];
#pragma unroll
  for (int q = 0; q < IPT; ++q) {
    const int e = q * T + threadIdx.x;
    rk[q] = e < tr.y ? L.rank[(size_t)tr.x + e] : NO_RANK;
  }
  __syncthreads();
#pragma unroll
  for (int b = 0; b < IPT; b += GB) {
    V4 ra[GB], rq[GB];
#pragma unroll
    for (int j = 0; j < GB; ++j) {
      if (rk[b + j] != NO_RANK) {
        const long long g = (long long)tr.x + (b + j) * T + threadIdx.x;
        ra[j] = rec[2 * g];
        rq[j] = rec[2 * g + 1];
      }
    }
#pragma unroll
    for (int j = 0; j < GB; ++j) {
      if (rk[b + j] == NO_RANK) continue;
      const uint32_t bn = th > 1 ? part_of(bin_key(ra[j].w), BM, tab) / PARTS : 0u;
      const long long dst = gb + L.bin_at[2 * t0 + bn] + rk[b + j];
      if (L.ms) ((R*)L.ms_b)[dst] = rq[j].w;
      put_binned(L, dst, ra[j], rq[j], (uint32_t)((long long)tr.x + (b + j) * T + threadIdx.x - gb));
    }
  }
}

// ---- segmented radix sort ------------------------------------------------------------

// Tile histograms, stored per halo digit-major: the count of digit d in the
// halo's tile i (i = t - t0) sits at hist[256 t0 + d T_h + i], T_h the halo's
// tile count, so each digit's column over the halo's tiles is contiguous.
template <typename Key>
__global__ void __launch_bounds__(T) g_hist(const Key* __restrict__ key, const int2* __restrict__ tile_range,
                                            const int* __restrict__ tile_halo, const int* __restrict__ halo_tile0,
                                            uint32_t* __restrict__ tile_hist, int shift) {
  __shared__ uint32_t h[256];
  const int t = blockIdx.x;
  const int2 tr = tile_range[t];
  const int k = tile_halo[t];
  const int t0 = halo_tile0[k], th = halo_tile0[k + 1] - t0;
  h[threadIdx.x] = 0;
  __syncthreads();
  for (int e = threadIdx.x; e < tr.y; e += T) atomicAdd(&h[(uint32_t)(key[tr.x + e] >> shift) & 0xffu], 1u);
  __syncthreads();
  tile_hist[(size_t)t0 * 256 + (size_t)threadIdx.x * th + (t - t0)] = h[threadIdx.x];
}

// Haloes of at most 256 tiles: one CTA per halo, thread d runs down digit
// d's column (exclusive prefix in place) and leaves the digit's total.
__global__ void __launch_bounds__(256) g_digit_scan_small(uint32_t* __restrict__ tile_hist,
                                                          const int* __restrict__ halo_tile0,
                                                          uint32_t* __restrict__ digit_base) {
  const int k = blockIdx.x, d = threadIdx.x;
  const int t0 = halo_tile0[k], th = halo_tile0[k + 1] - t0;
  if (th > 256) return;                  // g_digit_scan_big
  uint32_t* col = tile_hist + (size_t)t0 * 256 + (size_t)d * th;
  uint32_t run = 0;
  int i = 0;
  for (; i + 4 <= th; i += 4) {
    const uint32_t a = col[i], b = col[i + 1], c = col[i + 2], e = col[i + 3];
    col[i] = run;
    col[i + 1] = run + a;
    col[i + 2] = run + a + b;
    col[i + 3] = run + a + b + c;
    run += a + b + c + e;
  }
  for (; i < th; ++i) {
    const uint32_t a = col[i];
    col[i] = run;
    run += a;
  }
  digit_base[(size_t)k * 256 + d] = run;
}

// Haloes of more than 256 tiles: one CTA per (halo, digit) scans the column
// in chunks of 256 tiles.
__global__ void __launch_bounds__(256) g_digit_scan_big(uint32_t* __restrict__ tile_hist,
                                                        const int* __restrict__ halo_tile0,
                                                        const int* __restrict__ big, uint32_t* __restrict__ digit_base) {
  __shared__ uint32_t wt[8];
  __shared__ uint32_t carry;
  const int k = big[blockIdx.x >> 8], d = blockIdx.x & 255;
  const int t0 = halo_tile0[k], th = halo_tile0[k + 1] - t0;
  uint32_t* col = tile_hist + (size_t)t0 * 256 + (size_t)d * th;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int b = 0; b < th; b += 256) {
    const int i = b + threadIdx.x;
    const uint32_t v = i < th ? col[i] : 0u;
    const uint32_t inc = warp_inclusive_scan(v, lane);
    if (lane == 31) wt[warp] = inc;
    __syncthreads();
    uint32_t base = carry;
    for (int w = 0; w < warp; ++w) base += wt[w];
    if (i < th) col[i] = base + inc - v;
    __syncthreads();
    if (threadIdx.x == 255) carry = base + inc;
    __syncthreads();
  }
  if (threadIdx.x == 0) digit_base[(size_t)k * 256 + d] = carry;
}

// One CTA per halo: digit totals -> first destination of each digit.
__global__ void __launch_bounds__(256) g_digit_base(uint32_t* __restrict__ digit_base) {
  __shared__ uint32_t wt[8];
  const int k = blockIdx.x, d = threadIdx.x, lane = d & 31, warp = d >> 5;
  const uint32_t v = digit_base[(size_t)k * 256 + d];
  const uint32_t inc = warp_inclusive_scan(v, lane);
  if (lane == 31) wt[warp] = inc;
  __syncthreads();
  uint32_t base = inc - v;
  for (int w = 0; w < warp; ++w) base += wt[w];
  digit_base[(size_t)k * 256 + d] = base;
}

// Stable scatter of one tile by the digit at `shift`.  Each warp ranks its
// 8 batches of 32 keys by warp ballots on the digit's bits (the lanes with
// the same digit), the tile is re-ordered by digit in shared memory, and
// consecutive threads then write consecutive positions of each digit's run.
// FIRST: the values are the candidate positions (not read).  LAST: instead
// of (key, value) the radial-order streams are written from the records:
// (w, r), the mass (per-particle masses), u_th (gas) and the position; the
// tile's members' exact sum m v goes to tile_mv.
template <typename Key, typename R, bool FIRST, bool LAST>
__global__ void __launch_bounds__(T, LAST ? 3 : 5) g_scatter(GridLaunch L, const Key* __restrict__ kin,
                                               const uint32_t* __restrict__ vin, Key* __restrict__ kout,
                                               uint32_t* __restrict__ vout, int shift) {
  using V4 = typename Prec<R>::V4;
  using Acc = typename Prec<R>::Acc;
  __shared__ uint16_t whist[NWARP][256];
  __shared__ uint32_t dstart[256];
  __shared__ uint32_t gofs[256];
  __shared__ uint32_t red[NWARP];
  __shared__ Key skey[TILE];
  __shared__ uint32_t sval[TILE];
  const int t = blockIdx.x;
  const int2 tr = L.tile_range[t];
  const int kh = L.tile_halo[t];
  const long long gb = L.halos[kh].gbase;
  const int t0 = L.halo_tile0[kh], th = L.halo_tile0[kh + 1] - t0;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < NWARP * 256; i += T) (&whist[0][0])[i] = 0;
  // this tile's first global position of digit threadIdx.x (digit base + the
  // tiles before this one), loaded while the tile is ranked
  const uint32_t my_gofs =
      L.digit_base[(size_t)kh * 256 + threadIdx.x] + L.tile_hist[(size_t)t0 * 256 + (size_t)threadIdx.x * th + (t - t0)];
  constexpr int CH = TILE / NWARP;       // 256 elements per warp
  Key key[IPT];
  uint32_t val[IPT];
  uint16_t rank[IPT];
#pragma unroll
  for (int b = 0; b < IPT; ++b) {
    const int e = warp * CH + b * 32 + lane;
    const bool valid = e < tr.y;
    key[b] = valid ? kin[tr.x + e] : (Key)0;
    if (FIRST) val[b] = (uint32_t)((long long)tr.x + e - gb);
    else val[b] = valid ? vin[tr.x + e] : 0u;
  }
  __syncthreads();
#pragma unroll
  for (int b = 0; b < IPT; ++b) {
    const int e = warp * CH + b * 32 + lane;
    const bool valid = e < tr.y;
    const unsigned vmask = __ballot_sync(FULL_MASK, valid);
    const uint32_t dg = (uint32_t)(key[b] >> shift) & 0xffu;
    unsigned peers = vmask;
#pragma unroll
    for (int bit = 0; bit < 8; ++bit) {
      const unsigned bb = __ballot_sync(FULL_MASK, (dg >> bit) & 1u);
      peers &= ((dg >> bit) & 1u) ? bb : ~bb;
    }
    const unsigned below = peers & lanemask_lt();
    uint16_t base = 0;
    if (valid) base = whist[warp][dg];
    rank[b] = (uint16_t)(base + __popc(below));
    __syncwarp();
    if (valid && below == 0) whist[warp][dg] = (uint16_t)(base + __popc(peers));
    __syncwarp();
  }
  __syncthreads();
  {
    // per digit: offsets of each warp's run, the digit's start in the tile
    // and its first global position (digit base + tiles before this one)
    const int d = threadIdx.x;
    uint32_t run = 0;
#pragma unroll
    for (int w = 0; w < NWARP; ++w) {
      const uint32_t c = whist[w][d];
      whist[w][d] = (uint16_t)run;
      run += c;
    }
    dstart[d] = block_excl(run, red);
    gofs[d] = my_gofs;
  }
  __syncthreads();
#pragma unroll
  for (int b = 0; b < IPT; ++b) {
    const int e = warp * CH + b * 32 + lane;
    if (e < tr.y) {
      const uint32_t dg = (uint32_t)(key[b] >> shift) & 0xffu;
      const uint32_t lp = dstart[dg] + whist[warp][dg] + rank[b];
      skey[lp] = key[b];
      sval[lp] = val[b];
    }
  }
  __syncthreads();
  Acc smv[3] = {0, 0, 0};
  const int s_v = LAST ? L.state[kh].s_mv : 0;
  if (!LAST) {
    for (int i = threadIdx.x; i < tr.y; i += T) {
      const Key k = skey[i];
      const uint32_t dg = (uint32_t)(k >> shift) & 0xffu;
      const long long dst = gb + (long long)gofs[dg] + (i - (int)dstart[dg]);
      kout[dst] = k;
      vout[dst] = sval[i];
    }
  } else {
    // the records are gathered in batches of GB, every load of a batch issued
    // before its first use (the gathers are random within the halo)
    constexpr int GB = sizeof(R) == 4 ? 4 : 2;
    const V4* __restrict__ rec = (const V4*)L.rec;
#pragma unroll
    for (int b0 = 0; b0 < IPT; b0 += GB) {
      V4 ra[GB], rq[GB];
      uint32_t vv[GB];
      long long dd[GB];
      bool mem[GB];
#pragma unroll
      for (int j = 0; j < GB; ++j) {
        const int i = (b0 + j) * T + threadIdx.x;
        mem[j] = false;
        dd[j] = -1;
        if (i < tr.y) {
          const Key k = skey[i];
          vv[j] = sval[i];
          const uint32_t dg = (uint32_t)(k >> shift) & 0xffu;
          dd[j] = gb + (long long)gofs[dg] + (i - (int)dstart[dg]);
          mem[j] = k != ~(Key)0;
          if (mem[j]) {
            ra[j] = rec[2 * (gb + vv[j])];
            rq[j] = rec[2 * (gb + vv[j]) + 1];
          }
        }
      }
#pragma unroll
      for (int j = 0; j < GB; ++j) {
        if (dd[j] < 0) continue;
        const long long dst = dd[j];
        L.val_x[dst] = vv[j];
        if (!mem[j]) continue;
        const V4 a = ra[j], q = rq[j];
        ((V4*)L.wr)[dst] = a;
        if (L.ms) ((R*)L.ms)[dst] = q.w;
        if (L.uth) {
          const long long slot = L.halos[kh].offset + vv[j];
          const long long pi = L.out.member_idx ? L.out.member_idx[slot] : slot;
          ((R*)L.uth)[dst] = (R)(L.p.coord_type == AHF_COORD_F64 ? __ldg((const double*)L.p.u_th + pi)
                                                                 : (double)__ldg((const float*)L.p.u_th + pi));
        }
        smv[0] += fixr(mul_rn(q.w, q.x), s_v);
        smv[1] += fixr(mul_rn(q.w, q.y), s_v);
        smv[2] += fixr(mul_rn(q.w, q.z), s_v);
      }
    }
  }
  if (LAST) {
    __shared__ Acc racc[NWARP];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const Acc s = block_sum(smv[a], racc);
      if (threadIdx.x == 0) A<Acc>(L.tile_mv[3 * (size_t)t + a]) = s;
    }
  }
}

// No radix pass (every key equal): the radial order is the candidate order.
template <typename R>
__global__ void __launch_bounds__(T) g_fill_identity(GridLaunch L) {
  using V4 = typename Prec<R>::V4;
  using Key = typename Prec<R>::Key;
  using Acc = typename Prec<R>::Acc;
  const int t = blockIdx.x;
  const int2 tr = L.tile_range[t];
  const int kh = L.tile_halo[t];
  const long long gb = L.halos[kh].gbase;
  const int s_v = L.state[kh].s_mv;
  const Key* key = (const Key*)L.key_a;
  Acc smv[3] = {0, 0, 0};
  for (int e = threadIdx.x; e < tr.y; e += T) {
    const long long g = (long long)tr.x + e;
    const uint32_t v = (uint32_t)(g - gb);
    L.val_x[g] = v;
    if (key[g] != ~(Key)0) {
      const V4* rc = (const V4*)L.rec + 2 * g;
      const V4 a = rc[0], q = rc[1];
      ((V4*)L.wr)[g] = a;
      if (L.ms) ((R*)L.ms)[g] = q.w;
      if (L.uth) {
        const long long slot = L.halos[kh].offset + v;
        const long long pi = L.out.member_idx ? L.out.member_idx[slot] : slot;
        ((R*)L.uth)[g] = (R)(L.p.coord_type == AHF_COORD_F64 ? __ldg((const double*)L.p.u_th + pi)
                                                             : (double)__ldg((const float*)L.p.u_th + pi));
      }
      smv[0] += fixr(mul_rn(q.w, q.x), s_v);
      smv[1] += fixr(mul_rn(q.w, q.y), s_v);
      smv[2] += fixr(mul_rn(q.w, q.z), s_v);
    }
  }
  __shared__ Acc racc[NWARP];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const Acc s = block_sum(smv[a], racc);
    if (threadIdx.x == 0) A<Acc>(L.tile_mv[3 * (size_t)t + a]) = s;
  }
}

// ---- sub-tiles: the unit of a pass -------------------------------------------------------

// Sub-tile u covers elements [(u % SPT) SUB, (u % SPT + 1) SUB) of tile u / SPT
// (clipped to the tile); one warp handles it, element j of row i at position
// 32 i + lane, so that each row is one coalesced access.
constexpr int SUB = GRID_SUB;           // 256
constexpr int SPT = TILE / SUB;         // 8 sub-tiles per tile
constexpr int ROWS = SUB / 32;          // 8
constexpr int HT_BIG = 1024;            // threads of the per-halo kernel (largest halo > 64 tiles)
constexpr int HT_SMALL = 256;           // (otherwise)

// True once a pass of this call gave up waiting for a tensor copy: the
// sums it left are incomplete, so every later kernel of the class skips its
// work (the call's outputs are undefined and ahf_sync reports the timeout).
__device__ __forceinline__ bool gave_up(const GridLaunch& L) { return (__ldcg(L.out.err) & ERR_TIMEOUT) != 0; }

// Atomic add of an exact sum into a slot (the __int128 one from two 64-bit
// atomics: the low word's carry goes into the high word, so the total is
// exact once every addition has landed).
__device__ __forceinline__ void atomic_acc(AccSlot& s, long long v) {
  atomicAdd((unsigned long long*)&s.w[0], (unsigned long long)v);
}
__device__ __forceinline__ void atomic_acc(AccSlot& s, __int128 v) {
  const unsigned long long lo = (unsigned long long)v;
  const unsigned long long hi = (unsigned long long)((unsigned __int128)v >> 64);
  const unsigned long long old = atomicAdd((unsigned long long*)&s.w[0], lo);
  const unsigned long long carry = (old + lo < old) ? 1ull : 0ull;
  atomicAdd((unsigned long long*)&s.w[1], hi + carry);
}

// The same on a plain array of sums.
__device__ __forceinline__ void atomic_add_acc(long long* p, long long v) {
  atomicAdd((unsigned long long*)p, (unsigned long long)v);
}
__device__ __forceinline__ void atomic_add_acc(__int128* p, __int128 v) { atomic_acc(*(AccSlot*)p, v); }

// The map of a halo of one bin, from its own keys: 256 cells between the
// extreme keys, parts by the cells' counts.  `cell`: 256 zeroed words, left zero.
template <typename Key, int NE>
__device__ __forceinline__ BinMap one_bin_map(const Key key[NE], int n, uint32_t* cell, uint32_t* tab, uint32_t* red) {
  __shared__ uint32_t ext[2];
  __shared__ uint32_t total;
  if (threadIdx.x == 0) {
    ext[0] = 0x7f800000u;
    ext[1] = 0u;
  }
  __syncthreads();
  uint32_t a = 0x7f800000u, b = 0u;
#pragma unroll
  for (int j = 0; j < NE; ++j) {
    if (j * T + (int)threadIdx.x < n) {
      const uint32_t x = bin_key(radius_of_key(key[j]));
      a = min(a, x);
      b = max(b, x);
    }
  }
  a = __reduce_min_sync(FULL_MASK, a);
  b = __reduce_max_sync(FULL_MASK, b);
  if ((threadIdx.x & 31) == 0) {
    atomicMin(&ext[0], a);
    atomicMax(&ext[1], b);
  }
  __syncthreads();
  BinMap M;
  M.k0 = ext[0];
  M.kx = 0xffffffffu;                    // no tails
  M.tb = 0u;
  M.main = PARTS;
  M.cells = 256;
  const uint32_t range = ext[1] > ext[0] ? ext[1] - ext[0] : 0u;
  M.sh = max(0, 24 - __clz(max(range, 1u)));             // 256 << sh > range
  M.gs = 0;
#pragma unroll
  for (int j = 0; j < NE; ++j)
    if (j * T + (int)threadIdx.x < n) atomicAdd(&cell[(bin_key(radius_of_key(key[j])) - M.k0) >> M.sh], 1u);
  __syncthreads();
  const uint32_t w = 16u * cell[threadIdx.x] + 1u;
  cell[threadIdx.x] = 0u;
  const uint32_t base = block_excl(w, red);
  if (threadIdx.x == 255) total = base + w;
  __syncthreads();
  tab[threadIdx.x] = (PARTS * TAB_UNIT * base) / total;  // base <= 16 BIN_MAX + 256
  if (threadIdx.x == 0) tab[256] = PARTS * TAB_UNIT;
  __syncthreads();
  return M;
}

// v_bulk = sum m v / sum m of the current set, into the halo state.
template <typename R>
__device__ __forceinline__ void set_vbulk(GridHaloState& S, typename Prec<R>::Acc m,
                                          const typename Prec<R>::Acc mv[3]) {
  if (sizeof(R) == 4) {
    const float mt = from_fix(m, S.s_m, R());
    for (int a = 0; a < 3; ++a) S.vbulk[a] = (float)from_fix(mv[a], S.s_mv, R()) / mt;
  } else {
    const double mt = dfix(m, S.s_m);
    for (int a = 0; a < 3; ++a) S.vbulk_d[a] = dfix(mv[a], S.s_mv) / mt;
  }
}

// x 2^-s from an exact sum: in the mixed mode float_from_fix's bits, with
// 2^-s passed as a float (0 when it is not a normal float: then the general
// route); in the FP64 mode the nearest double.
__device__ __forceinline__ float fix_to_real(long long v, int s, float sc, float) {
  if (sc == 0.0f) return float_from_fix(v, s);
  const float hi = (float)(int)(v >> 32);
  const float lo = (float)(unsigned)(v & 0xffffffffll);
  return fmaf(hi, 4294967296.0f, lo) * sc;
}
__device__ __forceinline__ double fix_to_real(__int128 v, int s, float, double) { return double_from_fix128(v, s); }

// Sums of the initial set (all members alive) per sub-tile, one warp each,
// into copy 1 (the first pass's).
template <typename R>
__global__ void __launch_bounds__(T) g_sums(GridLaunch L) {
  using V4 = typename Prec<R>::V4;
  using Acc = typename Prec<R>::Acc;
  const int lane = threadIdx.x & 31;
  const int n_sub = L.n_tiles * SPT;
  const int u = (blockIdx.x * T + threadIdx.x) >> 5;     // one warp per sub-tile
  if (u >= n_sub) return;
  const V4* wr = (const V4*)L.wr;
  const R* ms = (const R*)L.ms;
  const R m0 = sizeof(R) == 4 ? (R)L.p.m0f : (R)L.p.m0;
  const int t = u / SPT;
  const int2 tr = L.tile_range[t];
  const int e0 = (u % SPT) * SUB;
  // the rows are read before the halo's state arrives (the loads depend on
  // the tile only); elements past the last member are dropped afterwards
  R rq[ROWS], mq[ROWS];
#pragma unroll
  for (int i = 0; i < ROWS; ++i) {
    const int e = e0 + 32 * i + lane;
    const long long g = (long long)tr.x + e;
    rq[i] = e < tr.y ? wr[g].w : (R)0;
    mq[i] = (e < tr.y && ms) ? ms[g] : m0;
  }
  const int k = L.tile_halo[t];
  const GridHaloState& S = L.state[k];
  const long long lim = L.halos[k].gbase + S.n_member;
  Acc a = 0, b = 0;
  int c = 0;
#pragma unroll
  for (int i = 0; i < ROWS; ++i) {
    const int e = e0 + 32 * i + lane;
    const long long g = (long long)tr.x + e;
    if (e < tr.y && g < lim) {
      a += fixp(mq[i], S.s_m);
      b += fixp(mq[i] * rinv_real(rq[i], L.prm), S.s_mr);
      ++c;
    }
  }
  a = wsum(a);
  b = wsum(b);
  c = __reduce_add_sync(FULL_MASK, c);
  if (lane == 0) {
    ((Acc*)L.agg_m)[n_sub + u] = a;
    ((Acc*)L.agg_r)[n_sub + u] = b;
    L.agg_c[n_sub + u] = c;
  }
}

// A halo's bookkeeping, by one thread, after the initial sums (INIT) or after
// pass `pass`: iterations, particle-iterations, band tests, sum m v, v_bulk,
// convergence (Sect. 2.1, Appendix A: the loop ends when an iteration removes
// nothing), from the sums M, Rr and the count C of the set left (mvs: sum m v of
// the members, INIT only).  Returns whether the halo goes on.
template <typename R, bool INIT>
__device__ __forceinline__ int halo_update(const GridLaunch& L, GridHaloState& S, int pass,
                                           typename Prec<R>::Acc M, typename Prec<R>::Acc Rr, long long C,
                                           const typename Prec<R>::Acc mvs[3], float vb[3]) {
  using Acc = typename Prec<R>::Acc;
  Acc mv[3];
  int active;
  if (INIT) {
#pragma unroll
    for (int q = 0; q < 3; ++q) mv[q] = mvs[q];
    active = C > 0 ? 1 : 0;
  } else {
    const long long alive = S.n_alive;
    S.part_iter += alive;
    S.band += S.band_pass;
    S.band_pass = 0;
    S.n_iter = pass;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      mv[q] = Ald<Acc>(S.mv[q]) - Ald<Acc>(S.rem_mv[q]);
      A<Acc>(S.rem_mv[q]) = 0;
    }
    active = 1;
    if (C == alive) {
      active = 0;
    } else if (C == 0) {
      active = 0;
      S.status |= AHF_HALO_EMPTY;
    } else if (pass >= L.prm.max_iter) {
      active = 0;
      S.status |= AHF_HALO_NOT_CONVERGED;
    }
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) A<Acc>(S.mv[q]) = mv[q];
  A<Acc>(S.m_tot) = M;
  A<Acc>(S.t_tot) = Rr;
  S.n_alive = C;
  if (active && (INIT || !L.prm.vbulk_initial)) set_vbulk<R>(S, M, mv);
  S.active = active;
  // the mass lost so far (exact sums), for the skip records and test
  if (INIT) A<Acc>(S.m_init) = M;
  S.mrem = INIT ? 0.0 : dfix(Ald<Acc>(S.m_init) - M, S.s_m);
#pragma unroll
  for (int q = 0; q < 3; ++q) vb[q] = sizeof(R) == 4 ? S.vbulk[q] : (float)S.vbulk_d[q];
  return active;
}

// Whether sub-tile u, last tested as `rc` says, may stay out of the next pass;
// if so its sums carry over to the copy that pass would have written.  It may
// while its members can neither be removed nor fall in the band: since that
// test each member's 2|phi| fell by at most 2 G dM / max(r, r_soft) (the halo
// lost mass dM, each removed particle's term at most m / r of the member's own
// radius), and its |u|^2 rose by at most 2 |u| dv + dv^2 (v_bulk moved by dv); the
// record's margin (slack 2^-16 of 2|phi| for the float rounding of both tests)
// must exceed that, with 2^-10 more on the bound for its own rounding.
template <typename R>
__device__ __forceinline__ bool skips(const GridLaunch& L, int u, int pass, const SkipRec& rc, double mrem, float vb0,
                                      float vb1, float vb2) {
  using Acc = typename Prec<R>::Acc;
  const float dm = (float)(mrem - rc.mrem) * (1.0f + 0x1p-20f);
  const float reff = fmaxf(rc.rin, L.prm.r_soft_f);
  const float ax = vb0 - rc.vb[0], ay = vb1 - rc.vb[1], az = vb2 - rc.vb[2];
  const float vmag =
      fabsf(vb0) + fabsf(vb1) + fabsf(vb2) + fabsf(rc.vb[0]) + fabsf(rc.vb[1]) + fabsf(rc.vb[2]);
  const float dv = sqrtf(fmaf(az, az, fmaf(ay, ay, ax * ax))) * (1.0f + 0x1p-20f) + vmag * 0x1p-20f;
  const float bound =
      ((2.0f * L.prm.Gf) * dm / reff + dv * fmaf(2.0f, rc.umax, dv)) * (1.0f + 0x1p-10f);
  if (!(reff > 0.0f && isfinite(bound) && rc.margin > bound)) return false;
  const size_t n_sub = (size_t)L.n_tiles * SPT;
  const size_t a = (size_t)((pass + 1) & 1) * n_sub + u, b = (size_t)(pass & 1) * n_sub + u;
  ((Acc*)L.agg_m)[b] = ((const Acc*)L.agg_m)[a];
  ((Acc*)L.agg_r)[b] = ((const Acc*)L.agg_r)[a];
  L.agg_c[b] = L.agg_c[a];
  return true;
}

// A halo of at most GRID_WARP_TILES tiles (32 sub-tiles), by one warp, a sub-tile per
// lane: g_halo's work without a CTA's barriers.  3,000 haloes in FP64 (2,900 of
// them this small) took 36 us a pass with one CTA each.
static_assert(GRID_WARP_TILES * SPT == 32, "a sub-tile per lane");
template <typename R, bool INIT>
__device__ __forceinline__ void halo_warp(const GridLaunch& L, int k, int pass) {
  using Acc = typename Prec<R>::Acc;
  GridHaloState& S = L.state[k];
  if (!INIT && !S.active) return;
  const int lane = threadIdx.x & 31;
  const int n_sub = L.n_tiles * SPT;
  const size_t cp = (size_t)((pass + 1) & 1) * n_sub;
  const int t0 = L.halo_tile0[k], th = L.halo_tile0[k + 1] - t0;
  const int u = t0 * SPT + lane;
  const long long nm = S.n_member;
  const int nu = (int)((nm + SUB - 1) / SUB);            // sub-tiles holding members
  SkipRec rc;
  if (!INIT && lane < nu) rc = L.skip[u];
  Acc m = 0, r = 0;
  int c = 0;
  if (lane < nu) {
    m = ((const Acc*)L.agg_m)[cp + u];
    r = ((const Acc*)L.agg_r)[cp + u];
    c = L.agg_c[cp + u];
  }
  const Acc im = wscan(m, lane), ir = wscan(r, lane);
  const int ic = (int)wscan((uint32_t)c, lane);
  if ((lane % SPT) == 0 && lane / SPT < th) {
    ((Acc*)L.pre_m)[t0 + lane / SPT] = im - m;
    ((Acc*)L.pre_r)[t0 + lane / SPT] = ir - r;
    L.pre_c[t0 + lane / SPT] = ic - c;
  }
  const Acc M = shfl_idx_x(im, 31), Rr = shfl_idx_x(ir, 31);
  const long long C = __shfl_sync(FULL_MASK, ic, 31);
  Acc mvs[3] = {0, 0, 0};
  if (INIT) {
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      if (lane < th) mvs[q] = Ald<Acc>(L.tile_mv[3 * (size_t)(t0 + lane) + q]);
      mvs[q] = wsum(mvs[q]);
    }
  }
  float vb[3] = {0.0f, 0.0f, 0.0f};
  int active = 0;
  double mrem = 0.0;
  if (lane == 0) {
    active = halo_update<R, INIT>(L, S, pass, M, Rr, C, mvs, vb);
    mrem = S.mrem;
  }
  active = __shfl_sync(FULL_MASK, active, 0);
  if (!active) return;
  mrem = __shfl_sync(FULL_MASK, mrem, 0);
#pragma unroll
  for (int q = 0; q < 3; ++q) vb[q] = __shfl_sync(FULL_MASK, vb[q], 0);
  bool keep = lane < nu;
  if (!INIT && keep && skips<R>(L, u, pass, rc, mrem, vb[0], vb[1], vb[2])) keep = false;
  const unsigned bal = __ballot_sync(FULL_MASK, keep);
  if (bal == 0u) {
    // every sub-tile left out: the next pass would remove nothing
    if (!INIT && lane == 0) {
      S.part_iter += S.n_alive;
      S.n_iter = pass + 1;
      S.active = 0;
    }
    return;
  }
  int base = 0;
  if (lane == 0) base = atomicAdd(&L.ctl->work_n[(pass + 1) & 1], __popc(bal));
  base = __shfl_sync(FULL_MASK, base, 0);
  if (keep) {
    int4* list = L.work + (size_t)((pass + 1) & 1) * n_sub;
    list[base + __popc(bal & lanemask_lt())] =
        make_int4(u, k, (int)(L.halos[k].gbase + (long long)lane * SUB), (int)min((long long)SUB, nm - (long long)lane * SUB));
  }
}

// Per halo, after the initial sums (INIT, pass 0) or after pass `pass`: the
// tiles' sums of the set left (copy (pass + 1) & 1 of the sub-tile sums),
// their exclusive prefix over the halo (for the next pass and the final one),
// the totals, and the halo's bookkeeping (halo_update).  Each thread takes a run
// of consecutive tiles; the runs' sums are scanned over the CTA.
// The sub-tiles of the haloes still active are listed for the next pass.
// The haloes are in order of size: the first L.n_cta_halos take a CTA each, the
// others (GRID_WARP_TILES tiles at most) a warp each.
template <typename R, bool INIT, int HT>
__global__ void __launch_bounds__(HT) g_halo(GridLaunch L, int pass) {
  if (gave_up(L)) return;
  using Acc = typename Prec<R>::Acc;
  constexpr int CH = 1024;                 // tiles per chunk held in shared memory
  constexpr int NW = HT / 32;
  __shared__ Acc racc[NW];
  __shared__ Acc wm_[NW], wr_[NW];
  __shared__ long long wc_[NW];
  __shared__ Acc tm_[CH], tr_[CH];
  __shared__ long long tc_[CH];
  __shared__ int s_nw;
  __shared__ Acc s_tm, s_tr;
  __shared__ long long s_tc;
  __shared__ float s_vb[3];                // the skip test's halo input
  __shared__ int s_wn[NW], s_wb[NW];       // kept sub-tiles per warp, their list positions
  __shared__ int s_kept;                   // sub-tiles of the halo on the next list
  if (INIT && bins_overflowed(L)) return;
  if (blockIdx.x >= L.n_cta_halos) {
    const int kw = L.n_cta_halos + (blockIdx.x - L.n_cta_halos) * NW + (threadIdx.x >> 5);
    if (kw < L.n_halos) halo_warp<R, INIT>(L, kw, pass);
    return;
  }
  const int k = blockIdx.x;
  GridHaloState& S = L.state[k];
  if (!INIT && !S.active) return;
  const int n_sub = L.n_tiles * SPT;
  const int cp = (pass + 1) & 1;
  const Acc* am = (const Acc*)L.agg_m + (size_t)cp * n_sub;
  const Acc* ar = (const Acc*)L.agg_r + (size_t)cp * n_sub;
  const int* ac = L.agg_c + (size_t)cp * n_sub;
  Acc* pm = (Acc*)L.pre_m;
  Acc* pr = (Acc*)L.pre_r;
  const int t0 = L.halo_tile0[k], t1 = L.halo_tile0[k + 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // only the sub-tiles holding members carry sums (the others are never
  // written by a pass)
  const int u_end = t0 * SPT + (int)((S.n_member + SUB - 1) / SUB);
  Acc cm = 0, cr = 0;                      // carry: the sums of the chunks before
  long long cc = 0;
  for (int c0 = t0; c0 < t1; c0 += CH) {
    const int cn = min(CH, t1 - c0);
    // tile sums, SPT lanes per tile (coalesced), reduced by shuffles; the
    // chunk's loads (CH * SPT / HT per thread) go out together
    constexpr int LPT = 8;
    for (int xr = 0; xr < cn * SPT; xr += LPT * HT) {
    Acc lm[LPT], lr[LPT];
    int lc[LPT];
#pragma unroll
    for (int q = 0; q < LPT; ++q) {
      const int x = xr + q * HT + threadIdx.x;
      const int u = c0 * SPT + x;
      const bool in = x < cn * SPT && u < u_end;
      lm[q] = in ? am[u] : (Acc)0;
      lr[q] = in ? ar[u] : (Acc)0;
      lc[q] = in ? ac[u] : 0;
    }
#pragma unroll
    for (int q = 0; q < LPT; ++q) {
      const int x = xr + q * HT + threadIdx.x;
      Acc m = lm[q], r = lr[q];
      int c = lc[q];
#pragma unroll
      for (int o = 1; o < SPT; o <<= 1) {
        m += shfl_xor_x(m, o);
        r += shfl_xor_x(r, o);
        c += shfl_xor_x(c, o);
      }
      if ((x % SPT) == 0 && x < cn * SPT) {
        tm_[x / SPT] = m;
        tr_[x / SPT] = r;
        tc_[x / SPT] = c;
      }
    }
    }
    __syncthreads();
    // exclusive scan of the chunk's tile sums: a run of consecutive tiles per thread
    const int per = (cn + HT - 1) / HT;
    const int j0 = min(cn, (int)threadIdx.x * per), j1 = min(j0 + per, cn);
    Acc sm = 0, sr = 0;
    long long sc = 0;
    for (int j = j0; j < j1; ++j) {
      sm += tm_[j];
      sr += tr_[j];
      sc += tc_[j];
    }
    const Acc im = wscan(sm, lane), ir = wscan(sr, lane);
    const long long ic = wscan(sc, lane);
    if (lane == 31) {
      wm_[warp] = im;
      wr_[warp] = ir;
      wc_[warp] = ic;
    }
    __syncthreads();
    if (warp == 0) {
      const bool in = lane < NW;
      const Acc xm = in ? wm_[lane] : (Acc)0, xr = in ? wr_[lane] : (Acc)0;
      const long long xc = in ? wc_[lane] : 0ll;
      const Acc ym = wscan(xm, lane), yr = wscan(xr, lane);
      const long long yc = wscan(xc, lane);
      __syncwarp();
      if (in) {
        wm_[lane] = ym - xm;
        wr_[lane] = yr - xr;
        wc_[lane] = yc - xc;
      }
      if (lane == 31) {
        s_tm = ym;
        s_tr = yr;
        s_tc = yc;
      }
    }
    __syncthreads();
    Acc em = cm + wm_[warp] + im - sm, er = cr + wr_[warp] + ir - sr;
    long long ec = cc + wc_[warp] + ic - sc;
    for (int j = j0; j < j1; ++j) {
      pm[c0 + j] = em;
      pr[c0 + j] = er;
      L.pre_c[c0 + j] = ec;
      em += tm_[j];
      er += tr_[j];
      ec += tc_[j];
    }
    cm += s_tm;
    cr += s_tr;
    cc += s_tc;
    __syncthreads();                       // the chunk's shared arrays are reused
  }
  const Acc M = cm, Rr = cr;
  const long long C = cc;
  Acc mvs[3] = {0, 0, 0};
  if (INIT) {
    // sum m v of the members, from the sort's per-tile sums
    for (int j = t0 + threadIdx.x; j < t1; j += HT)
#pragma unroll
      for (int q = 0; q < 3; ++q) mvs[q] += Ald<Acc>(L.tile_mv[3 * (size_t)j + q]);
#pragma unroll
    for (int q = 0; q < 3; ++q) mvs[q] = block_sum_n<Acc, HT>(mvs[q], racc);
  }
  if (threadIdx.x == 0) {
    const int active = halo_update<R, INIT>(L, S, pass, M, Rr, C, mvs, s_vb);
    // the halo's sub-tiles holding members go on the next pass's list
    s_nw = active ? (int)((S.n_member + SUB - 1) / SUB) : 0;
    s_kept = 0;
  }
  __syncthreads();
  const int nw = s_nw;
  if (nw) {
    const long long nm = S.n_member, gb = L.halos[k].gbase;
    int* wn = &L.ctl->work_n[(pass + 1) & 1];
    int4* list = L.work + (size_t)((pass + 1) & 1) * n_sub;
    const double mrem = S.mrem;
    const float vb0 = s_vb[0], vb1 = s_vb[1], vb2 = s_vb[2];
    // RB sub-tiles per thread and round, their records loaded together
    constexpr int RB = 4;
    for (int j0 = 0; j0 < nw; j0 += RB * HT) {
      bool keep[RB];
      SkipRec rc[RB];
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        const int j = j0 + r * HT + threadIdx.x;
        keep[r] = j < nw;
        if (!INIT && keep[r]) rc[r] = L.skip[t0 * SPT + j];
      }
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        const int j = j0 + r * HT + threadIdx.x;
        const int u = t0 * SPT + j;
        if (INIT || !keep[r]) continue;
        if (skips<R>(L, u, pass, rc[r], mrem, vb0, vb1, vb2)) keep[r] = false;
      }
      // list positions: a warp scan of the warps' counts, one reservation per round
      unsigned bal[RB];
      int cnt = 0;
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        bal[r] = __ballot_sync(FULL_MASK, keep[r]);
        cnt += __popc(bal[r]);
      }
      if (lane == 0) s_wn[warp] = cnt;
      __syncthreads();
      if (warp == 0) {
        const int x = lane < NW ? s_wn[lane] : 0;
        const int inc = (int)wscan((uint32_t)x, lane);
        int base = 0;
        if (lane == 31 && inc) base = atomicAdd(wn, inc);
        base = __shfl_sync(FULL_MASK, base, 31);
        if (lane < NW) s_wb[lane] = base + inc - x;
        if (lane == 31) s_kept += inc;
      }
      __syncthreads();
      int off = s_wb[warp];
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        const int j = j0 + r * HT + threadIdx.x;
        if (keep[r])
          list[off + __popc(bal[r] & lanemask_lt())] =
              make_int4(t0 * SPT + j, k, (int)(gb + (long long)j * SUB), (int)min((long long)SUB, nm - (long long)j * SUB));
        off += __popc(bal[r]);
      }
      __syncthreads();                     // s_wn, s_wb are reused
    }
    // every sub-tile left out: the next pass would remove nothing, so the
    // halo converges there (its particle-iterations counted, no band tests)
    if (!INIT && threadIdx.x == 0 && s_kept == 0) {
      S.part_iter += S.n_alive;
      S.n_iter = pass + 1;
      S.active = 0;
    }
  }
}

// The n members of a bin in order of (r, candidate position), for one in which a
// part holds more than PART_MAX: a bitonic sort in shared memory with every
// comparator pointing up, so that positions behind n need no padding.  78 rounds at
// most, bound by their barriers.  Leaving such a bin to the radix sort instead sent
// every halo of the call there, after the passes of a chunk without an active halo.
template <typename Key>
__device__ __noinline__ void order_tied(Key* skey, uint16_t* sidx, uint32_t* spos, int n) {
  auto order = [&](int lo, int hi) {     // lo < hi
    if (hi >= n) return;
    const Key a = skey[lo], b = skey[hi];
    const uint32_t p = spos[lo], q = spos[hi];
    if (a < b || (a == b && p < q)) return;
    const uint16_t x = sidx[lo];
    skey[lo] = b;
    skey[hi] = a;
    spos[lo] = q;
    spos[hi] = p;
    sidx[lo] = sidx[hi];
    sidx[hi] = x;
  };
  for (int half = 1; half < n; half <<= 1) {
    // mirrored pairs of each block of 2 half, then pairs at distance d
    for (int t = threadIdx.x; 2 * half * (t / half) + t % half < n; t += T) {
      const int at = 2 * half * (t / half);
      order(at + t % half, at + 2 * half - 1 - t % half);
    }
    __syncthreads();
    for (int d = half >> 1; d > 0; d >>= 1) {
      for (int t = threadIdx.x; 2 * d * (t / d) + t % d < n; t += T) {
        const int at = 2 * d * (t / d) + t % d;
        order(at, at + d);
      }
      __syncthreads();
    }
  }
}

// A bin ordered, one CTA each: its members counted in the bin's 512 parts in
// shared memory, their keys moved there, and each member's place in its part
// found by counting the members before it in (r, candidate).  Then, in
// radial order, the streams (w, r), (v, 1/r), the position (and mass, thermal
// energy), the exact sum m v, and the sub-tiles' sums of the initial set.
template <typename R>
__global__ void __launch_bounds__(T, sizeof(R) == 4 ? 4 : 3) g_bin_sort(GridLaunch L) {
  using V4 = typename Prec<R>::V4;
  using Key = typename Prec<R>::Key;
  using Acc = typename Prec<R>::Acc;
  constexpr int NE = BIN_MAX / T;        // members per thread
  extern __shared__ __align__(16) unsigned char dyn[];
  Key* skey = reinterpret_cast<Key*>(dyn);                       // [BIN_MAX]
  uint16_t* sidx = reinterpret_cast<uint16_t*>(skey + BIN_MAX);  // [BIN_MAX] slot -> source
  uint16_t* sout = sidx + BIN_MAX;                               // [BIN_MAX] place -> source
  uint16_t* spart = sout + BIN_MAX;                              // [BIN_MAX] slot -> part
  uint32_t* spos = reinterpret_cast<uint32_t*>(sout);            // order_tied: candidate positions
  __shared__ uint32_t tab[CELLS + 1];
  __shared__ uint32_t pcnt[PARTS + 1];
  __shared__ uint32_t red[NWARP];
  __shared__ Acc racc[NWARP];
  if (bins_overflowed(L)) return;
  const int bin = blockIdx.x, t = bin >> 1;
  const int k = L.tile_halo[t];
  const HaloDev& H = L.halos[k];
  const GridHaloState& S = L.state[k];
  const int t0 = L.halo_tile0[k], th = L.halo_tile0[k + 1] - t0;
  if (th == 1 && (bin & 1)) return;      // one bin
  const int n = (int)L.bin_n[(size_t)bin * BIN_PAD];
  BinMap BM;
  if (th > 1) BM = load_bin_map(L, k, t0, H.count, th, tab);
  pcnt[threadIdx.x] = 0u;
  pcnt[threadIdx.x + T] = 0u;
  Acc smv[3] = {0, 0, 0};
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t at = L.bin_at[bin];
  const long long g0 = H.gbase + at;     // first flat position of the bin
  const V4* __restrict__ rb = (const V4*)L.rec_b + 2 * g0;
  uint32_t slot[NE];                     // part << 16 | rank of arrival in it
  {
    Key key[NE];
#pragma unroll
    for (int j = 0; j < NE; ++j) {
      if (j * T >= n) break;
      const int i = j * T + threadIdx.x;
      if (i < n) key[j] = key_of(rb[2 * i].w);
    }
    __syncthreads();
    if (th == 1) BM = one_bin_map<Key, NE>(key, n, pcnt, tab, red);
    const uint32_t first = (uint32_t)PARTS * (uint32_t)(bin - 2 * t0);
#pragma unroll
    for (int j = 0; j < NE; ++j) {
      if (j * T >= n) break;
      const int i = j * T + threadIdx.x;
      if (i < n) {
        const uint32_t q = min(part_of(bin_key(radius_of_key(key[j])), BM, tab) - first, (uint32_t)PARTS - 1u);
        slot[j] = (q << 16) | atomicAdd(&pcnt[q], 1u);
      }
    }
    __syncthreads();
    const uint32_t v0 = pcnt[2 * threadIdx.x], v1 = pcnt[2 * threadIdx.x + 1];
    // (one way for the whole CTA)
    if (__syncthreads_or(max(v0, v1) > PART_MAX)) {
#pragma unroll
      for (int j = 0; j < NE; ++j) {
        const int i = j * T + threadIdx.x;
        if (i < n) {
          skey[i] = key[j];
          sidx[i] = (uint16_t)i;
          spos[i] = binned_pos(rb[2 * i + 1].w);
        }
      }
      __syncthreads();
      order_tied(skey, sidx, spos, n);
      for (int q = threadIdx.x; q < n; q += T) sout[q] = sidx[q];
    } else {
      const uint32_t ex = block_excl(v0 + v1, red);
      __syncthreads();
      pcnt[2 * threadIdx.x] = ex;
      pcnt[2 * threadIdx.x + 1] = ex + v0;
      if (threadIdx.x == T - 1) pcnt[PARTS] = ex + v0 + v1;
      __syncthreads();
#pragma unroll
      for (int j = 0; j < NE; ++j) {
        if (j * T >= n) break;
        const int i = j * T + threadIdx.x;
        if (i < n) {
          const uint32_t q = pcnt[slot[j] >> 16] + (slot[j] & 0xffffu);
          skey[q] = key[j];
          sidx[q] = (uint16_t)i;
          spart[q] = (uint16_t)(slot[j] >> 16);
        }
      }
      __syncthreads();
      // in slot order: a warp's members are in neighbouring parts
      for (int own = threadIdx.x; own < n; own += T) {
        const uint32_t p = spart[own];
        const uint32_t a = pcnt[p], z = pcnt[p + 1];
        const Key mine = skey[own];
        uint32_t q = a, ties = 0u;
        for (uint32_t x = a; x < z; ++x) {
          const Key kx = skey[x];
          q += kx < mine ? 1u : 0u;
          ties += kx == mine ? 1u : 0u;
        }
        const uint32_t ip = sidx[own];
        if (ties > 1u) {                 // equal radii: in candidate order
          const uint32_t pos = binned_pos(rb[2 * ip + 1].w);
          for (uint32_t x = a; x < z; ++x)
            if (skey[x] == mine && binned_pos(rb[2 * (uint32_t)sidx[x] + 1].w) < pos) ++q;
        }
        sout[q] = (uint16_t)ip;
      }
    }
  }
  __syncthreads();
  // the streams in radial order, a warp taking rows of 32; sums by sub-tile
  const int s_m = S.s_m, s_r = S.s_mr, s_v = S.s_mv;
  const R m0 = sizeof(R) == 4 ? (R)L.p.m0f : (R)L.p.m0;
  const Acc mfix0 = fixp(m0, s_m);
  V4* vr = (V4*)L.vr;
  const size_t sub0 = (size_t)L.n_tiles * SPT + (size_t)t0 * SPT;   // copy 1
  // rows aligned to 32 positions of the halo, so that none straddles two sub-tiles
  const int lead = (int)(at & 31u);
  const int rows = (n + lead + 31) >> 5;
  // each warp a run of rows: its lanes keep the sums of a sub-tile (8 rows) and
  // reduce them where it ends (144e6 members: 3.27 -> 3.17 ms with add_fix)
  const int share = (rows + NWARP - 1) / NWARP;
  const int row1 = min(rows, (warp + 1) * share);
  Acc a = 0, b = 0;
  int c = 0;
  for (int row = warp * share; row < row1; ++row) {
    const int e = row * 32 - lead + lane;
    const bool in = e >= 0 && e < n;
    if (in) {
      const int i = sout[e];
      const V4 x = rb[2 * i];
      V4 y = rb[2 * i + 1];
      const uint32_t p = binned_pos(y.w);
      const long long dst = g0 + e;
      const R m = L.ms ? ((const R*)L.ms_b)[g0 + i] : m0;
      const R ri = rinv_real(x.w, L.prm);
      y.w = ri;                          // (the mass is in ms, or uniform)
      ((V4*)L.wr)[dst] = x;
      vr[dst] = y;
      L.val_x[dst] = p;
      if (L.ms) ((R*)L.ms)[dst] = m;
      if (L.uth) {
        const long long slot = H.offset + p;
        const long long pi = L.out.member_idx ? L.out.member_idx[slot] : slot;
        ((R*)L.uth)[dst] = (R)(L.p.coord_type == AHF_COORD_F64 ? __ldg((const double*)L.p.u_th + pi)
                                                               : (double)__ldg((const float*)L.p.u_th + pi));
      }
      if (L.ms) add_fix(a, m, s_m);
      add_fix(b, m * ri, s_r);
      add_fix(smv[0], mul_rn(m, y.x), s_v);
      add_fix(smv[1], mul_rn(m, y.y), s_v);
      add_fix(smv[2], mul_rn(m, y.z), s_v);
    }
    c += __popc(__ballot_sync(FULL_MASK, in));
    const uint32_t u = (at - (uint32_t)lead + (uint32_t)row * 32u) / SUB;
    if (row + 1 == row1 || (at - (uint32_t)lead + (uint32_t)row * 32u + 32u) / SUB != u) {
      const Acc am = L.ms ? wsum(a) : mfix0 * (Acc)c, br = wsum(b);
      if (lane == 0 && c) {
        atomic_add_acc((Acc*)L.agg_m + sub0 + u, am);
        atomic_add_acc((Acc*)L.agg_r + sub0 + u, br);
        atomicAdd(&L.agg_c[sub0 + u], c);
      }
      a = 0;
      b = 0;
      c = 0;
    }
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const Acc x = block_sum(smv[a], racc);
    if (threadIdx.x == 0) atomic_acc(L.tile_mv[3 * (size_t)t + a], x);
  }
}

// ---- one unbinding pass -----------------------------------------------------------------

constexpr int EPL = SUB / 32;            // 8 consecutive elements per lane

// Prefix sums of a sub-tile's start: the tile's prefix plus the sums of the
// tile's sub-tiles before it in copy `cp` (lanes < u % SPT read one each).  With
// one mass for all (UNIF) M is the count times its fixed-point value mfix0.
template <bool UNIF, typename Acc>
__device__ __forceinline__ void sub_prefix(const GridLaunch& L, int u, int t, int cp, Acc mfix0, Acc& M, Acc& P,
                                           long long* C) {
  const int lane = threadIdx.x & 31;
  const int n_sub = L.n_tiles * SPT;
  const int ui = u % SPT;
  Acc m = 0, r = 0;
  int c = 0;
  if (lane < ui) {
    const size_t j = (size_t)cp * n_sub + (u - ui) + lane;
    if (!UNIF) m = ((const Acc*)L.agg_m)[j];
    r = ((const Acc*)L.agg_r)[j];
    if (UNIF || C) c = L.agg_c[j];
  }
  P = ((const Acc*)L.pre_r)[t] + wsum(r);
  long long n = 0;
  if (UNIF || C) n = L.pre_c[t] + __reduce_add_sync(FULL_MASK, c);
  if (UNIF) M = (Acc)n * mfix0;
  else M = ((const Acc*)L.pre_m)[t] + wsum(m);
  if (C) *C = n;
}

// The skip record of sub-tile u from the lanes' margins and |u|^2 maxima
// (lane 0's first element is the sub-tile's first: its |r| bounds the
// members' radii from below); conservative roundings to float.
template <typename R>
__device__ __forceinline__ void write_skip(const GridLaunch& L, int u, const GridHaloState& S, R mg, R uu, R r0,
                                           const R vb[3]) {
  // floats in order as integers (no NaN among them, |u|^2 not negative)
  int m, w;
  if (sizeof(R) == 4) {
    m = __float_as_int((float)mg);
    w = __float_as_int((float)uu);
  } else {
    m = __float_as_int(__double2float_rd((double)mg));
    w = __float_as_int(__double2float_ru((double)uu));
  }
  m = __reduce_min_sync(FULL_MASK, m ^ ((m >> 31) & 0x7fffffff));
  w = __reduce_max_sync(FULL_MASK, w);
  if ((threadIdx.x & 31) != 0) return;
  SkipRec rc;
  rc.margin = __int_as_float(m ^ ((m >> 31) & 0x7fffffff));
  rc.umax = __fsqrt_ru(__int_as_float(w));
  rc.rin = sizeof(R) == 4 ? fabsf((float)r0) : __double2float_rd(fabs((double)r0));
#pragma unroll
  for (int a = 0; a < 3; ++a) rc.vb[a] = (float)vb[a];
  rc.mrem = S.mrem;
  L.skip[u] = rc;
}

// The particles a pass removed from sub-tile w.x (flags `rem` of the lane's
// elements, nrem > 0 in the warp): the sign bit of r, their removal iteration, and
// the exact sum m v of what the halo lost.  They are listed in shared memory first
// (256 bytes a warp) and taken one per lane: a few of a sub-tile's 256 are removed,
// mostly by a few lanes.
template <typename R, bool UNIF>
__device__ __forceinline__ void removed(const GridLaunch& L, const int4 w, int pass, unsigned rem, int nrem, uint8_t* list) {
  using V4 = typename Prec<R>::V4;
  using Acc = typename Prec<R>::Acc;
  const int lane = threadIdx.x & 31;
  GridHaloState& S = L.state[w.y];
  const HaloDev& H = L.halos[w.y];
  V4* wr = (V4*)L.wr;
  const uint32_t n = (uint32_t)__popc(rem);
  uint32_t at = wscan(n, lane) - n;
  for (; rem; rem &= rem - 1) list[at++] = (uint8_t)(lane * EPL + __ffs(rem) - 1);
  __syncwarp();
  const R m0 = sizeof(R) == 4 ? (R)L.p.m0f : (R)L.p.m0;
  const int s_v = S.s_mv;
  Acc mv[3] = {0, 0, 0};
  for (int j = lane; j < nrem; j += 32) {
    const long long g = (long long)w.z + list[j];
    const uint32_t pos = L.val_x[g];
    const R m = UNIF ? m0 : ((const R*)L.ms)[g];
    // radial order, or (radix sort) the candidate's record
    const V4 v = L.vr ? ((const V4*)L.vr)[g] : ((const V4*)L.rec)[2 * (H.gbase + pos) + 1];
    if (sizeof(R) == 4) atomicOr((unsigned*)&wr[g].w, 0x80000000u);
    else atomicOr((unsigned long long*)&wr[g].w, 0x8000000000000000ull);
    if (L.out.removed_iter) L.out.removed_iter[H.offset + pos] = pass;
    add_fix(mv[0], mul_rn(m, v.x), s_v);
    add_fix(mv[1], mul_rn(m, v.y), s_v);
    add_fix(mv[2], mul_rn(m, v.z), s_v);
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    mv[a] = wsum(mv[a]);
    if (lane == 0) atomic_acc(S.rem_mv[a], mv[a]);
  }
  __syncwarp();                          // the list is reused
}

// 2 |phi|: -2 phi_real, the doubling (exact) in the factor.
__device__ __forceinline__ float two_phi_real(float M, float ri, float S, const ParamsDev& P) {
  return -2.0f * phi_real(M, ri, S, P);
}
__device__ __forceinline__ double two_phi_real(double M, double ri, double S, const ParamsDev& P) {
  return __dmul_rn(2.0 * P.G, __fma_rn(M, ri, S));
}

// The escape and band tests of a member and the skip record's extremes (the
// smallest margin and the largest |u|^2 of the members kept; NaN left out).
template <typename R>
struct BandTest {
  R band, mg = (R)INFINITY, uu = (R)0;
  __device__ __forceinline__ explicit BandTest(R b) : band(b) {}
  __device__ __forceinline__ bool in_band(R u2, R two_phi) const { return fabs(u2 - two_phi) < band * two_phi; }
  __device__ __forceinline__ bool escapes(R u2, R two_phi) const { return u2 > two_phi; }
  __device__ __forceinline__ void keep(R margin, R uk) {
    mg = fmin(mg, margin);
    uu = fmax(uu, uk);
  }
  __device__ __forceinline__ void extremes(R& m, R& u) const {
    m = mg;
    u = uu;
  }
};
// In FP64 on the integer pipe: the bit patterns of positive doubles compare as
// they do, two within band (< 1/4) of each other differ by less than band 2^54
// in them, and the extremes are kept as upper words (rounded down and up at
// the end: the skip test is one-sided).  A member takes 10 FP64 instructions (44
// with the division, the comparisons and the conversions).
template <>
struct BandTest<double> {
  double band;
  unsigned long long near;               // differences of the bits that may be in the band
  int mg = 0x7ff00000, uu = -1;
  __device__ __forceinline__ explicit BandTest(double b) : band(b) {
    near = b >= 0.0 && b < 0.25 ? (unsigned long long)(b * 0x1p54) + 2ull : ~0ull;
  }
  static __device__ __forceinline__ bool plain(unsigned long long a, unsigned long long b) {
    return a <= INF_BITS && b <= INF_BITS;
  }
  __device__ __forceinline__ bool in_band(double u2, double two_phi) const {
    const unsigned long long a = (unsigned long long)__double_as_longlong(u2);
    const unsigned long long b = (unsigned long long)__double_as_longlong(two_phi);
    if (plain(a, b) && (a > b ? a - b : b - a) > near) return false;
    return fabs(u2 - two_phi) < band * two_phi;
  }
  __device__ __forceinline__ bool escapes(double u2, double two_phi) const {
    const unsigned long long a = (unsigned long long)__double_as_longlong(u2);
    const unsigned long long b = (unsigned long long)__double_as_longlong(two_phi);
    return plain(a, b) ? a > b : u2 > two_phi;
  }
  __device__ __forceinline__ void keep(double margin, double uk) {
    const int h = __double2hiint(margin), w = __double2hiint(uk);
    mg = min(mg, (h & 0x7fffffff) > 0x7ff00000 ? 0x7ff00000 : h ^ ((h >> 31) & 0x7fffffff));
    uu = max(uu, w > 0x7ff00000 ? -1 : w);
  }
  __device__ __forceinline__ void extremes(double& m, double& u) const {
    // (upper words in order, the lower ones dropped: one down for negative
    // margins, one up for |u|^2)
    const int o = mg < 0 ? mg - 1 : mg;
    m = __hiloint2double(o ^ ((o >> 31) & 0x7fffffff), 0);
    u = uu < 0 ? 0.0 : __hiloint2double(min(uu + 1, 0x7ff00000), 0);
  }
};

// Phi and the escape test over sub-tile w.x (halo w.y) in pass `pass`, by
// one warp: lane l holds elements [8 l, 8 l + 8) of the sub-tile; one warp
// scan of the lanes' sums places every element's prefix.  It leaves the
// sub-tile's sums after the removals for the next pass and marks the removed
// (a kernel of its own for that cost 6 to 60 us a pass).
// FAST: the scales 2^-s of the halo are normal floats (the conversions of
// the exact sums to float are then a multiply; same bits).
template <typename R, bool UNIF, bool GAS, bool FAST>
__device__ __forceinline__ void pass_sub(const GridLaunch& L, const int4 w, int pass, uint8_t* list) {
  using V4 = typename Prec<R>::V4;
  using Acc = typename Prec<R>::Acc;
  const int u = w.x, k = w.y, t = u / SPT;
  GridHaloState& S = L.state[k];
  const int lane = threadIdx.x & 31;
  const int s_m = S.s_m, s_r = S.s_mr;
  const ParamsDev& P = L.prm;
  const int n_sub = L.n_tiles * SPT;
  const int cp = pass & 1;
  const long long gl = (long long)w.z + lane * EPL;   // the lane's first element
  const int nl = w.w - lane * EPL;                    // its members (<= 0: none)
  const V4* wr = (const V4*)L.wr;
  const R m0 = sizeof(R) == 4 ? (R)L.p.m0f : (R)L.p.m0;
  // the lane's elements, all in flight at once
  V4 q[EPL];
  R mq[EPL], uq[EPL], ri[EPL];
  // FP64: 1/r as the bins' sort left it beside v (a division is a third of the
  // FP64 instructions of a member)
  const bool has_ri = sizeof(R) == 8 && L.vr != nullptr;
#pragma unroll
  for (int i = 0; i < EPL; ++i) {
    const long long g = gl + i;
    ri[i] = (R)0;
    if (i < nl) {
      q[i] = wr[g];
      if (has_ri) ri[i] = ((const V4*)L.vr)[g].w;
      mq[i] = UNIF ? m0 : ((const R*)L.ms)[g];
      uq[i] = GAS ? ((const R*)L.uth)[g] : (R)0;
    } else {
      q[i].x = q[i].y = q[i].z = (R)0;
      q[i].w = neg0(R());
      mq[i] = m0;
      uq[i] = (R)0;
    }
  }
  const Acc mfix0 = fixp(m0, s_m);
  Acc M, Pp;
  sub_prefix<UNIF>(L, u, t, cp, mfix0, M, Pp, nullptr);
  R vb[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) vb[a] = sizeof(R) == 4 ? (R)S.vbulk[a] : (R)S.vbulk_d[a];
  const R band = sizeof(R) == 4 ? (R)P.band_f : (R)P.band;
  const Acc Ttot = Ald<Acc>(S.t_tot);
  const float sc_m = FAST ? pow2_neg(s_m) : 0.0f, sc_r = FAST ? pow2_neg(s_r) : 0.0f;
  // per element: 1/r and the exact terms; the lane's sums
  Acc rf[EPL];
  Acc a = 0, b = 0;
  uint32_t na = 0;
#pragma unroll
  for (int i = 0; i < EPL; ++i) {
    const bool alive = !signbit(q[i].w);
    if (!has_ri) ri[i] = rinv_real(q[i].w, P);
    rf[i] = alive ? fixp(mq[i] * ri[i], s_r) : (Acc)0;
    if (UNIF) na += alive ? 1u : 0u;
    else if (alive) a += fixp(mq[i], s_m);
    b += rf[i];
  }
  if (UNIF) M += (Acc)(wscan(na, lane) - na) * mfix0;
  else M += wscan(a, lane) - a;
  Pp += wscan(b, lane) - b;
  const size_t jc = (size_t)cp * n_sub + u;
  const Acc n_m = ((const Acc*)L.agg_m)[jc], n_r = ((const Acc*)L.agg_r)[jc];
  const int n_c = L.agg_c[jc];
  // phi and the escape test; the skip record's margin and |u| over the
  // members left alive
  unsigned rem = 0;
  int nband = 0;
  Acc rm = 0, rr = 0;
  const R keep_frac = (R)1 - band - (R)0x1p-16;
  R mg = (R)INFINITY, uu = (R)0;
  BandTest<R> test(band);
#pragma unroll
  for (int i = 0; i < EPL; ++i) {
    const R r = q[i].w;
    if (!signbit(r)) {
      const Acc mfix = UNIF ? mfix0 : fixp(mq[i], s_m);
      const R Mf = (FAST && sizeof(R) == 4) ? (R)fix_to_float_sc((long long)M, sc_m) : from_fix(M, s_m, R());
      const R Sf = (FAST && sizeof(R) == 4) ? (R)fix_to_float_sc((long long)(Ttot - Pp), sc_r)
                                            : from_fix(Ttot - Pp, s_r, R());
      const R two_phi = two_phi_real(Mf, ri[i], Sf, P);
      const R ux = q[i].x - vb[0], uy = q[i].y - vb[1], uz = q[i].z - vb[2];
      const R uk = fma_x(uz, uz, fma_x(uy, uy, ux * ux));
      R u2 = uk;
      if (GAS) u2 += (R)2 * uq[i];                 // gas: |u|^2 + 2 u_th (Sect. 2.1)
      if (test.in_band(u2, two_phi)) ++nband;
      if (test.escapes(u2, two_phi)) {
        rem |= 1u << i;
        rm += mfix;
        rr += rf[i];
      } else {
        test.keep(fma_x(two_phi, keep_frac, -u2), uk);
      }
      M += mfix;
      Pp += rf[i];
    }
  }
  test.extremes(mg, uu);
  write_skip<R>(L, u, S, mg, uu, q[0].w, vb);
  // the sub-tile's sums after the removals (next copy) and its removal flags
  const int nrem = __reduce_add_sync(FULL_MASK, __popc(rem));
  nband = __reduce_add_sync(FULL_MASK, nband);
  if (nrem) {                                      // uniform over the warp
    rm = wsum(rm);
    rr = wsum(rr);
    removed<R, UNIF>(L, w, pass, rem, nrem, list);
  }
  if (lane == 0) {
    const size_t j = (size_t)(cp ^ 1) * n_sub + u;
    ((Acc*)L.agg_m)[j] = n_m - rm;
    ((Acc*)L.agg_r)[j] = n_r - rr;
    L.agg_c[j] = n_c - nrem;
    if (nband) atomicAdd((unsigned long long*)&S.band_pass, (unsigned long long)nband);
  }
}

// One pass: warps take the listed sub-tiles (those of the active haloes)
// round robin, and clear the count of the next pass's list.
// PER: CTAs an SM.  In FP64 one (211 registers, nothing spilt) while that gives
// every sub-tile its warp, else two (128 registers): 3,000 haloes 1268 -> 1214 us
// with two, one halo of 43 sub-tiles 266 us with one and 274 with two.
template <typename R, bool UNIF, bool GAS, int PER>
__global__ void __launch_bounds__(T, PER) g_pass(GridLaunch L, int pass) {
  __shared__ uint8_t removed_list[NWARP][SUB];
  if (blockIdx.x == 0 && threadIdx.x == 0) L.ctl->work_n[(pass + 1) & 1] = 0;
  if (gave_up(L)) return;
  const int n = __ldcg(&L.ctl->work_n[pass & 1]);
  const int4* list = L.work + (size_t)(pass & 1) * L.n_tiles * SPT;
  for (int i = (blockIdx.x * T + threadIdx.x) >> 5; i < n; i += (gridDim.x * T) >> 5) {
    const int4 w = list[i];
    const GridHaloState& S = L.state[w.y];
    if (sizeof(R) == 4 && pow2_neg(S.s_m) != 0.0f && pow2_neg(S.s_mr) != 0.0f)
      pass_sub<R, UNIF, GAS, true>(L, w, pass, removed_list[threadIdx.x >> 5]);
    else
      pass_sub<R, UNIF, GAS, false>(L, w, pass, removed_list[threadIdx.x >> 5]);
  }
}

// ---- the pass with tensor copies into shared memory (mixed mode) -----------------------

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// One 4 KB box (32 rows of 8 elements) of the stream into dst; bar counts it.
__device__ __forceinline__ void tma_box(void* dst, const CUtensorMap* map, int row, uint64_t* bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], 4096;" ::"r"(smem_u32(bar)) : "memory");
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(map), "r"(0), "r"(row), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t phase) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(phase)
      : "memory");
  return ok != 0;
}
// Wait for a barrier phase with at most `limit` polls; false if it gave up.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t phase, long long limit) {
  for (long long i = 0; i < limit; ++i)
    if (mbar_test(bar, phase)) return true;
  return false;
}
constexpr long long DRAIN_POLLS = 1ll << 24;   // a warp that gave up still lets its copies land

// Element i of lane `lane` of a box copied with the 128-byte swizzle: row
// `lane`, 16-byte chunk i stored at chunk i ^ (lane & 7).
__device__ __forceinline__ float4 box_at(const float4* box, int lane, int i) { return box[lane * 8 + (i ^ (lane & 7))]; }

// One sub-tile from its box in shared memory (the mixed mode, a uniform
// particle mass, no gas): the arithmetic of pass_sub.
template <bool FAST>
__device__ __forceinline__ void pass_box(const GridLaunch& L, const int4 w, int pass, const float4* box, uint8_t* list) {
  using Acc = long long;
  const int u = w.x, k = w.y, t = u / SPT;
  GridHaloState& S = L.state[k];
  const int lane = threadIdx.x & 31;
  const int s_m = S.s_m, s_r = S.s_mr;
  const ParamsDev& P = L.prm;
  const int n_sub = L.n_tiles * SPT;
  const int cp = pass & 1;
  const int nl = w.w - lane * EPL;                    // the lane's members (<= 0: none)
  const float m0 = L.p.m0f;
  const Acc mfix0 = fixp(m0, s_m);
  Acc M, Pp;
  sub_prefix<true>(L, u, t, cp, mfix0, M, Pp, nullptr);
  const float vb0 = S.vbulk[0], vb1 = S.vbulk[1], vb2 = S.vbulk[2];
  const float band = P.band_f;
  const Acc Ttot = Ald<Acc>(S.t_tot);
  const float sc_m = FAST ? pow2_neg(s_m) : 0.0f, sc_r = FAST ? pow2_neg(s_r) : 0.0f;
  float ri[EPL];
  Acc rf[EPL];
  Acc b = 0;
  unsigned alive = 0;
#pragma unroll
  for (int i = 0; i < EPL; ++i) {
    const float r = box_at(box, lane, i).w;
    const bool al = i < nl && !signbit(r);
    alive |= (al ? 1u : 0u) << i;
    ri[i] = rinv_real(r, P);
    rf[i] = al ? fixp(m0 * ri[i], s_r) : 0ll;
    b += rf[i];
  }
  const uint32_t na = (uint32_t)__popc(alive);
  M += (Acc)(wscan(na, lane) - na) * mfix0;
  Pp += wscan(b, lane) - b;
  const size_t jc = (size_t)cp * n_sub + u;
  const Acc n_m = ((const Acc*)L.agg_m)[jc], n_r = ((const Acc*)L.agg_r)[jc];
  const int n_c = L.agg_c[jc];
  unsigned rem = 0;
  int nband = 0;
  Acc rr = 0;
  const float keep_frac = 1.0f - band - 0x1p-16f;
  float mg = INFINITY, uu = 0.0f;
#pragma unroll
  for (int i = 0; i < EPL; ++i) {
    if (alive & (1u << i)) {
      const float4 q = box_at(box, lane, i);
      const float Mf = FAST ? fix_to_float_sc(M, sc_m) : float_from_fix(M, s_m);
      const float Sf = FAST ? fix_to_float_sc(Ttot - Pp, sc_r) : float_from_fix(Ttot - Pp, s_r);
      const float phi = phi_of(Mf, ri[i], Sf, P.Gf);
      const float ux = q.x - vb0, uy = q.y - vb1, uz = q.z - vb2;
      const float u2 = fmaf(uz, uz, fmaf(uy, uy, ux * ux));
      const float two_phi = -2.0f * phi;
      if (fabsf(u2 - two_phi) < band * two_phi) ++nband;
      if (u2 > two_phi) {
        rem |= 1u << i;
        rr += rf[i];
      } else {
        mg = fminf(mg, fmaf(two_phi, keep_frac, -u2));
        uu = fmaxf(uu, u2);
      }
      M += mfix0;
      Pp += rf[i];
    }
  }
  {
    const float vbv[3] = {vb0, vb1, vb2};
    write_skip<float>(L, u, S, mg, uu, box_at(box, lane, 0).w, vbv);
  }
  const int nrem = __reduce_add_sync(FULL_MASK, __popc(rem));
  nband = __reduce_add_sync(FULL_MASK, nband);
  if (nrem) {
    rr = wsum(rr);
    removed<float, true>(L, w, pass, rem, nrem, list);
  }
  if (lane == 0) {
    const size_t j = (size_t)(cp ^ 1) * n_sub + u;
    ((Acc*)L.agg_m)[j] = n_m - (Acc)nrem * mfix0;
    ((Acc*)L.agg_r)[j] = n_r - rr;
    L.agg_c[j] = n_c - nrem;
    if (nband) atomicAdd((unsigned long long*)&S.band_pass, (unsigned long long)nband);
  }
}

// One pass with the sub-tiles streamed into shared memory by tensor copies:
// each warp keeps two 4 KB boxes, fetching its next sub-tile while it
// computes the current one.  Waits are bounded by L.wait_limit polls; a warp
// that gives up sets ERR_TIMEOUT, lets its copies land and stops.
constexpr int TMA_SMEM = NWARP * 2 * 4096 + NWARP * 2 * 8;
__global__ void __launch_bounds__(T, 3) g_pass_tma(const __grid_constant__ GridLaunch L, int pass) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ uint8_t removed_list[NWARP][SUB];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float4* box0 = (float4*)(smem + warp * 8192);
  uint64_t* bar = (uint64_t*)(smem + NWARP * 8192) + 2 * warp;
  if (blockIdx.x == 0 && threadIdx.x == 0) L.ctl->work_n[(pass + 1) & 1] = 0;
  if (gave_up(L)) return;
  const int n = __ldcg(&L.ctl->work_n[pass & 1]);
  const int4* list = L.work + (size_t)(pass & 1) * L.n_tiles * SPT;
  const int stride = gridDim.x * NWARP;
  int i = blockIdx.x * NWARP + warp;
  if (i >= n) return;
  if (smem_u32(smem) & 1023) {                       // the swizzled boxes need 1 KB alignment
    if (lane == 0) atomicOr(L.out.err, ERR_TIMEOUT);
    return;
  }
  if (lane == 0) {
    mbar_init(&bar[0]);
    mbar_init(&bar[1]);
    fence_async_smem();
  }
  __syncwarp();
  uint32_t phase0 = 0, phase1 = 0;
  int4 w = list[i];
  if (lane == 0) tma_box(box0, &L.wr_map, w.z >> 3, &bar[0]);
  for (int b = 0; i < n; i += stride, b ^= 1) {
    const int inext = i + stride;
    const int4 wn = inext < n ? list[inext] : make_int4(0, 0, 0, 0);
    __syncwarp();
    if (inext < n && lane == 0) {
      fence_async_smem();
      tma_box(box0 + (b ^ 1) * 256, &L.wr_map, wn.z >> 3, &bar[b ^ 1]);
    }
    const uint32_t ph = b ? phase1 : phase0;
    if (!mbar_wait(&bar[b], ph, L.wait_limit)) {
      if (lane == 0) atomicOr(L.out.err, ERR_TIMEOUT);
      mbar_wait(&bar[b], ph, DRAIN_POLLS);
      if (inext < n) mbar_wait(&bar[b ^ 1], b ? phase0 : phase1, DRAIN_POLLS);
      return;
    }
    if (b) phase1 ^= 1;
    else phase0 ^= 1;
    const GridHaloState& S = L.state[w.y];
    if (pow2_neg(S.s_m) != 0.0f && pow2_neg(S.s_mr) != 0.0f) pass_box<true>(L, w, pass, box0 + b * 256, removed_list[warp]);
    else pass_box<false>(L, w, pass, box0 + b * 256, removed_list[warp]);
    w = wn;
  }
}

// ---- final pass --------------------------------------------------------------------------

// Bound lists (radial order), phi of the final set, compacted radius and
// inclusive mass for the virial search and the profile rows; one warp per
// sub-tile, lanes holding consecutive elements as in a pass.
template <typename R, bool UNIF>
__global__ void __launch_bounds__(T, sizeof(R) == 4 ? 4 : 2) g_final(GridLaunch L) {
  if (gave_up(L)) return;
  using V4 = typename Prec<R>::V4;
  using Acc = typename Prec<R>::Acc;
  const int lane = threadIdx.x & 31;
  const int n_sub = L.n_tiles * SPT;
  const int u = (blockIdx.x * T + threadIdx.x) >> 5;     // one warp per sub-tile
  if (u >= n_sub) return;
  const V4* wr = (const V4*)L.wr;
  R* rc = (R*)L.rc;
  Acc* mc = (Acc*)L.mc;
  const R m0 = sizeof(R) == 4 ? (R)L.p.m0f : (R)L.p.m0;
  const ParamsDev& P = L.prm;
  const int t = u / SPT;
  const int2 tr = L.tile_range[t];
  const int e0 = (u % SPT) * SUB;
  // rows of 32 consecutive elements (coalesced), read before the halo's
  // state arrives; elements past the last member count as removed
  R rq[ROWS], mq[ROWS], ri_q[ROWS];
  uint32_t vq[ROWS];
  const bool has_ri = sizeof(R) == 8 && L.vr != nullptr;   // as in a pass
#pragma unroll
  for (int i = 0; i < ROWS; ++i) {
    const int e = e0 + 32 * i + lane;
    const long long g = (long long)tr.x + e;
    rq[i] = e < tr.y ? wr[g].w : neg0(R());
    mq[i] = (!UNIF && e < tr.y) ? ((const R*)L.ms)[g] : m0;
    ri_q[i] = has_ri && e < tr.y ? ((const V4*)L.vr)[g].w : (R)0;
    vq[i] = e < tr.y ? L.val_x[g] : 0u;
  }
  const int k = L.tile_halo[t];
  const GridHaloState& S = L.state[k];
  if (S.n_alive == 0) return;
  const HaloDev& H = L.halos[k];
  const long long lim = H.gbase + S.n_member;
  const int s_m = S.s_m, s_r = S.s_mr;
  const Acc Ttot = Ald<Acc>(S.t_tot);
  Acc M, Pp;
  long long C;
  const Acc mfix0 = fixp(m0, s_m);
  sub_prefix<UNIF>(L, u, t, (S.n_iter + 1) & 1, mfix0, M, Pp, &C);
  const float sc_m = pow2_neg(s_m), sc_r = pow2_neg(s_r);
  const unsigned below = lanemask_lt();
#pragma unroll
  for (int i = 0; i < ROWS; ++i) {
    const R r = rq[i];
    const bool alive = !signbit(r) && (long long)tr.x + e0 + 32 * i + lane < lim;
    const R ri = has_ri ? ri_q[i] : rinv_real(r, P);
    const Acc a = UNIF || !alive ? (Acc)0 : (Acc)fixp(mq[i], s_m);
    const Acc b = alive ? (Acc)fixp(mq[i] * ri, s_r) : (Acc)0;
    const unsigned bal = __ballot_sync(FULL_MASK, alive);
    if (bal == 0u) continue;
    const Acc ia = UNIF ? (Acc)0 : wscan(a, lane), ib = wscan(b, lane);
    if (alive) {
      // M(<r) before the particle, and the outer sum from the particle out
      const Acc Mi = UNIF ? M + (Acc)__popc(bal & below) * mfix0 : M + ia - a;
      const R phi = phi_real(fix_to_real(Mi, s_m, sc_m, R()), ri,
                             fix_to_real(Ttot - (Pp + ib - b), s_r, sc_r, R()), P);
      const long long slot = H.offset + vq[i];
      const long long pi = L.out.member_idx ? L.out.member_idx[slot] : slot;
      const long long c = C + __popc(bal & below);
      L.out.bound_idx[H.offset + c] = pi;
      if (L.out.phi) ((R*)L.out.phi)[H.offset + c] = phi;
      rc[H.gbase + c] = r;
      if (!UNIF) mc[H.gbase + c] = M + ia;     // (uniform: the rank times the mass)
    }
    if (UNIF) M += (Acc)__popc(bal) * mfix0;
    else M += shfl_idx_x(ia, 31);
    Pp += shfl_idx_x(ib, 31);
    C += __popc(bal);
  }
}

// First compacted index k with M_k < delta_rho 4pi/3 r_{k+1}^3 (r_{N+1} = inf).
template <typename R>
__global__ void __launch_bounds__(T) g_virial(GridLaunch L) {
  if (gave_up(L)) return;
  using Acc = typename Prec<R>::Acc;
  const R* rc = (const R*)L.rc;
  const Acc* mc = (const Acc*)L.mc;
  const int t = blockIdx.x;
  const int k = L.tile_halo[t];
  GridHaloState& S = L.state[k];
  const int2 tr = L.tile_range[t];
  const long long gb = L.halos[k].gbase;
  const long long nb = S.n_alive;
  const ParamsDev& P = L.prm;
  const bool unif = L.ms == nullptr;
  const Acc mfix0 = fixp(sizeof(R) == 4 ? (R)L.p.m0f : (R)L.p.m0, S.s_m);
  long long kf = 0x7fffffffffffffffll;
  for (int e = threadIdx.x; e < tr.y; e += T) {
    const long long g = (long long)tr.x + e;
    const long long kk = g - gb;
    if (kk >= nb) break;
    bool cross = true;
    if (kk + 1 < nb) {
      const Acc mk = unif ? (Acc)(kk + 1) * mfix0 : mc[g];
      if (sizeof(R) == 4) {
        const float rn = (float)rc[g + 1];
        const float lhs = from_fix(mk, S.s_m, R());
        const float rhs = P.crit_f * rn * rn * rn;
        if (lhs < rhs * (1.0f - 1e-5f)) cross = true;
        else if (lhs > rhs * (1.0f + 1e-5f)) cross = false;
        else {
          const double rd = (double)rn;
          cross = dfix(mk, S.s_m) < P.crit * rd * rd * rd;
        }
      } else {
        const double rd = (double)rc[g + 1];
        const double mkd = L.p.m == nullptr ? (double)(kk + 1) * L.p.m0 : dfix(mk, S.s_m);
        cross = mkd < P.crit * rd * rd * rd;
      }
    }
    if (cross) {
      kf = kk;
      break;
    }
  }
  for (int o = 16; o > 0; o >>= 1) kf = min(kf, __shfl_xor_sync(FULL_MASK, kf, o));
  if ((threadIdx.x & 31) == 0 && kf != 0x7fffffffffffffffll)
    atomicMin((unsigned long long*)&S.k_first, (unsigned long long)kf);
}

template <typename R>
__global__ void g_result(GridLaunch L) {
  if (gave_up(L)) return;
  using Acc = typename Prec<R>::Acc;
  const R* rc = (const R*)L.rc;
  const Acc* mcv = (const Acc*)L.mc;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= L.n_halos) return;
  const GridHaloState& S = L.state[k];
  const HaloDev& H = L.halos[k];
  ahf_result Rs;
  const long long nb = S.n_alive;
  Rs.n_bound = nb;
  Rs.n_member = S.n_member;
  Rs.part_iter = S.part_iter;
  Rs.n_band = S.band;
  Rs.n_iter = S.n_iter;
  Rs.k_vir = -1;
  Rs.m_vir = 0.0;
  Rs.r_vir = 0.0;
  int status = S.status;
  if (S.n_member == 0) status |= AHF_HALO_EMPTY;
  if (nb > 0) {
    const long long kk = S.k_first;
    // M_vir: (k+1) m0 in FP64 for a uniform mass, else the exact sum
    const bool unim = L.p.m == nullptr;
    const Acc mkx = unim ? (Acc)0 : mcv[H.gbase + kk];
    const double mk = unim ? double_from_fix(kk + 1, 0) * L.p.m0 : dfix(mkx, S.s_m);
    if (kk == nb - 1) status |= AHF_HALO_RVIR_BEYOND_EDGE;
    bool none;
    if (sizeof(R) == 4) {
      // the decision and the values as in the on-chip classes (the same bits)
      const float mkf = unim ? (float)(kk + 1) * L.p.m0f : (float)from_fix(mkx, S.s_m, R());
      none = below_threshold(mk, mkf, (float)rc[H.gbase + kk], L.prm.crit_f, L.prm.crit);
    } else {
      const double rk = (double)rc[H.gbase + kk];
      none = mk < L.prm.crit * rk * rk * rk;
    }
    if (none) {
      status |= AHF_HALO_RVIR_NONE;
    } else {
      Rs.k_vir = kk;
      Rs.m_vir = mk;
      Rs.r_vir = virial_radius(mk, L.prm.inv_crit);
      if (L.prm.rise_edge && kk == nb - 1) {
        auto at = [&](long long j, double& r, double& m) {
          r = sizeof(R) == 4 ? float_to_double((float)rc[H.gbase + j]) : (double)rc[H.gbase + j];
          m = unim ? double_from_fix(j + 1, 0) * L.p.m0 : dfix(mcv[H.gbase + j], S.s_m);
        };
        const long long ke = rise_edge_index(nb, at);
        if (ke >= 0) {
          at(ke, Rs.r_vir, Rs.m_vir);
          Rs.k_vir = ke;
          status |= AHF_HALO_RISE_EDGE;
        }
      }
    }
    const double mt = dfix(Ald<Acc>(S.m_tot), S.s_m);
    for (int a = 0; a < 3; ++a) Rs.vbulk[a] = quotient(dfix(Ald<Acc>(S.mv[a]), S.s_mv), mt);
  } else {
    Rs.vbulk[0] = Rs.vbulk[1] = Rs.vbulk[2] = 0.0;
  }
  Rs.status = status;
  L.out.res[H.index] = Rs;
}

// Profile rows of every halo of the class from its compacted bound set (one
// CTA per halo, the rows spread over the threads; Sect. 2.1's radially binned
// output): each edge by binary search over the compacted radii.
__global__ void __launch_bounds__(T) g_rows_mixed(GridLaunch L) {
  if (gave_up(L)) return;
  const int k = blockIdx.x;
  const HaloDev& H = L.halos[k];
  const GridHaloState& S = L.state[k];
  const ahf_result& Rs = L.out.res[H.index];
  const double m0 = L.p.m0;
  const long long gb = H.gbase;
  profile_rows(L.rows, H.index, (const float*)L.rc, (const long long*)L.mc, [gb](long long j) { return gb + j; },
               S.n_alive, Rs.r_vir, Rs.k_vir, S.s_m, L.prm.G, L.prm.Gf, L.p.m == nullptr ? &m0 : nullptr, threadIdx.x, T);
}

// The all-FP64 rows: FP64 radii against the FP64 edges, __int128 masses.
__global__ void __launch_bounds__(T) g_rows_f64(GridLaunch L) {
  if (gave_up(L)) return;
  const int k = blockIdx.x;
  const HaloDev& H = L.halos[k];
  const GridHaloState& S = L.state[k];
  const ahf_result& Rs = L.out.res[H.index];
  const ProfileRows& Q = L.rows;
  const int n = Q.n_bins;
  double* out = Q.prof + (size_t)H.index * n * 4;
  const long long nb = S.n_alive;
  const double* rc = (const double*)L.rc + H.gbase;
  const __int128* mc = (const __int128*)L.mc + H.gbase;
  if (nb == 0) {
    for (int i = threadIdx.x; i < 4 * n; i += T) out[i] = 0.0;
    return;
  }
  const double r_out = Rs.r_vir > 0.0 ? Rs.r_vir : rc[nb - 1];
  const float inv_r = 1.0f / double_to_float(r_out);
  auto count_le = [&](int b) {               // first j with rc[j] > e_b (b = n: r_out)
    const double e = b == n ? r_out : r_out * Q.factor[b];
    long long lo = 0, hi = nb;
    while (lo < hi) {
      const long long mid = (lo + hi) >> 1;
      if (rc[mid] <= e) lo = mid + 1;
      else hi = mid;
    }
    return lo;
  };
  for (int b = threadIdx.x; b < n; b += T) {
    const long long c0 = count_le(b), c1 = count_le(b + 1);
    double M1, Mshell;
    if (L.p.m == nullptr) {
      M1 = double_from_fix(c1, 0) * L.p.m0;
      Mshell = double_from_fix(c1 - c0, 0) * L.p.m0;
    } else {
      const __int128 f0 = c0 > 0 ? mc[c0 - 1] : (__int128)0;
      const __int128 f1 = c1 > 0 ? mc[c1 - 1] : (__int128)0;
      M1 = double_from_fix128(f1, S.s_m);
      Mshell = double_from_fix128(f1 - f0, S.s_m);
    }
    out[4 * b + 0] = double_from_fix(c1 - c0, 0);
    out[4 * b + 1] = M1;
    out[4 * b + 2] = shell_density(Mshell, r_out, inv_r, Q.factor, Q.factor_f, n, b);
    out[4 * b + 3] = circular_velocity(L.prm.G, L.prm.Gf, M1, r_out, inv_r, Q.factor, Q.factor_f, n, b);
  }
}

inline int blocks_for(int n, int b) { return (n + b - 1) / b; }

template <typename R, bool BINS>
void launch_prepare(const GridLaunch& L, cudaStream_t s) {
  const bool f64 = L.p.coord_type == AHF_COORD_F64;
  if constexpr (sizeof(R) == 4) {
    if (f64) g_prepare_mixed<AHF_COORD_F64, BINS><<<L.n_tiles, T, 0, s>>>(L);
    else g_prepare_mixed<AHF_COORD_F32_REL, BINS><<<L.n_tiles, T, 0, s>>>(L);
  } else {
    if (f64) g_prepare_f64<AHF_COORD_F64, BINS><<<L.n_tiles, T, 0, s>>>(L);
    else g_prepare_f64<AHF_COORD_F32_REL, BINS><<<L.n_tiles, T, 0, s>>>(L);
  }
}

// CTAs of g_halo: one per large halo, then one warp per small one.
int halo_ctas(const GridLaunch& L, int threads) {
  return L.n_cta_halos + blocks_for(L.n_halos - L.n_cta_halos, threads / 32);
}

template <typename R>
void launch_halo_init(const GridLaunch& L, cudaStream_t s) {
  if (L.max_halo_tiles > 64) g_halo<R, true, HT_BIG><<<halo_ctas(L, HT_BIG), HT_BIG, 0, s>>>(L, 0);
  else g_halo<R, true, HT_SMALL><<<halo_ctas(L, HT_SMALL), HT_SMALL, 0, s>>>(L, 0);
}

// The distribution into radial bins (see g_sample).
template <typename R>
cudaError_t bins_t(GridLaunch& L, cudaStream_t s) {
  L.sort_launches = 0;
  if (L.n_tiles == 0) {
    g_scales<R><<<blocks_for(L.n_halos, 128), 128, 0, s>>>(L);
    L.sort_launches = 1;
    return cudaGetLastError();
  }
  constexpr size_t smem = (size_t)BIN_MAX * (sizeof(typename Prec<R>::Key) + 6);
  static std::atomic<unsigned long long> attrs_set{0};
  cudaError_t e = cudaSuccess;
  if (first_use_on_device(attrs_set)) {
    e = cudaFuncSetAttribute(g_bin_sort<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    mark_used_on_device(attrs_set);
  }
  if (L.max_halo_tiles > 1) {
    const int shares = std::min(L.max_halo_tiles, SAMPLE_MAX / T);
    const bool by_halo = L.n_halos > 1 && L.n_halos <= 65535 && (long long)shares * L.n_halos < L.n_tiles;
    const dim3 grid = by_halo ? dim3((unsigned)shares, (unsigned)L.n_halos) : dim3((unsigned)L.n_tiles);
    if (L.p.coord_type == AHF_COORD_F64) g_sample<R, AHF_COORD_F64><<<grid, T, 0, s>>>(L);
    else g_sample<R, AHF_COORD_F32_REL><<<grid, T, 0, s>>>(L);
    g_bin_map<<<L.n_halos, SAMPLE_T, 0, s>>>(L);
  }
  launch_prepare<R, true>(L, s);
  g_bin_base<R><<<L.n_halos, T, 0, s>>>(L);
  g_place<R><<<L.n_tiles, T, 0, s>>>(L);
  g_bin_sort<R><<<2 * L.n_tiles, T, smem, s>>>(L);
  launch_halo_init<R>(L, s);
  L.sort_launches = 5 + (L.max_halo_tiles > 1 ? 2 : 0);
  return cudaGetLastError();
}

template <typename R>
cudaError_t prepare_t(const GridLaunch& L, cudaStream_t s) {
  if (L.n_tiles > 0) launch_prepare<R, false>(L, s);
  g_scales<R><<<blocks_for(L.n_halos, 128), 128, 0, s>>>(L);
  return cudaGetLastError();
}

template <typename R>
cudaError_t sort_t(GridLaunch& L, cudaStream_t s, unsigned long long or_bits, unsigned long long and_bits) {
  using Key = typename Prec<R>::Key;
  const unsigned long long diff = or_bits ^ and_bits;
  int digits[8];
  int nd = 0;
  for (int d = 0; d < (int)sizeof(Key); ++d)
    if ((diff >> (8 * d)) & 0xffull) digits[nd++] = d;
  if (L.n_tiles == 0) nd = 0;
  L.sort_launches = 0;
  if (L.n_tiles == 0) return cudaGetLastError();
  Key *ki = (Key*)L.key_a, *ko = (Key*)L.key_b;
  uint32_t *vi = L.val_a, *vo = L.val_b;
  for (int p = 0; p < nd; ++p) {
    const int shift = 8 * digits[p];
    // the prepare left the low byte's tile counts
    if (p > 0 || shift != 0) {
      g_hist<Key><<<L.n_tiles, T, 0, s>>>(ki, L.tile_range, L.tile_halo, L.halo_tile0, L.tile_hist, shift);
      ++L.sort_launches;
    }
    L.sort_launches += 3 + (L.n_big ? 1 : 0);
    g_digit_scan_small<<<L.n_halos, 256, 0, s>>>(L.tile_hist, L.halo_tile0, L.digit_base);
    if (L.n_big) g_digit_scan_big<<<L.n_big * 256, 256, 0, s>>>(L.tile_hist, L.halo_tile0, L.big_halos, L.digit_base);
    g_digit_base<<<L.n_halos, 256, 0, s>>>(L.digit_base);
    const bool first = p == 0, last = p == nd - 1;
    if (first && last) g_scatter<Key, R, true, true><<<L.n_tiles, T, 0, s>>>(L, ki, vi, ko, vo, shift);
    else if (first) g_scatter<Key, R, true, false><<<L.n_tiles, T, 0, s>>>(L, ki, vi, ko, vo, shift);
    else if (last) g_scatter<Key, R, false, true><<<L.n_tiles, T, 0, s>>>(L, ki, vi, ko, vo, shift);
    else g_scatter<Key, R, false, false><<<L.n_tiles, T, 0, s>>>(L, ki, vi, ko, vo, shift);
    Key* x = ki;
    ki = ko;
    ko = x;
    uint32_t* y = vi;
    vi = vo;
    vo = y;
  }
  if (nd == 0) g_fill_identity<R><<<L.n_tiles, T, 0, s>>>(L);
  L.sort_launches += (nd == 0 ? 1 : 0) + 2;
  g_sums<R><<<(int)(((long long)L.n_tiles * SPT + NWARP - 1) / NWARP), T, 0, s>>>(L);
  launch_halo_init<R>(L, s);
  return cudaGetLastError();
}

std::atomic<unsigned long long> g_tma_attr{0};

template <typename R, int PER>
void launch_pass(const GridLaunch& L, int pass, int grid, cudaStream_t s) {
  const bool unif = L.ms == nullptr, gas = L.uth != nullptr;
  if (unif && !gas) g_pass<R, true, false, PER><<<grid, T, 0, s>>>(L, pass);
  else if (!unif && !gas) g_pass<R, false, false, PER><<<grid, T, 0, s>>>(L, pass);
  else if (unif) g_pass<R, true, true, PER><<<grid, T, 0, s>>>(L, pass);
  else g_pass<R, false, true, PER><<<grid, T, 0, s>>>(L, pass);
}

template <typename R>
cudaError_t iterate_t(const GridLaunch& L, int pass, cudaStream_t s) {
  const bool unif = L.ms == nullptr, gas = L.uth != nullptr;
  if (sizeof(R) == 4 && L.use_tma && unif && !gas) {
    if (first_use_on_device(g_tma_attr)) {
      const cudaError_t e = cudaFuncSetAttribute(g_pass_tma, cudaFuncAttributeMaxDynamicSharedMemorySize, TMA_SMEM);
      if (e != cudaSuccess) return e;
      mark_used_on_device(g_tma_attr);
    }
    g_pass_tma<<<L.tma_grid, T, TMA_SMEM, s>>>(L, pass);
  } else if constexpr (sizeof(R) == 4) {
    launch_pass<R, 2>(L, pass, L.iter_grid, s);
  } else if ((long long)L.n_tiles * SPT > (long long)L.iter_grid * NWARP) {
    launch_pass<R, 2>(L, pass, 2 * L.iter_grid, s);
  } else {
    launch_pass<R, 1>(L, pass, L.iter_grid, s);
  }
  if (L.max_halo_tiles > 64) g_halo<R, false, HT_BIG><<<halo_ctas(L, HT_BIG), HT_BIG, 0, s>>>(L, pass);
  else g_halo<R, false, HT_SMALL><<<halo_ctas(L, HT_SMALL), HT_SMALL, 0, s>>>(L, pass);
  return cudaGetLastError();
}

template <typename R>
cudaError_t finish_t(const GridLaunch& L, cudaStream_t s) {
  if (L.n_tiles > 0) {
    const int nb = (int)(((long long)L.n_tiles * SPT + NWARP - 1) / NWARP);
    if (L.ms == nullptr) g_final<R, true><<<nb, T, 0, s>>>(L);
    else g_final<R, false><<<nb, T, 0, s>>>(L);
    g_virial<R><<<L.n_tiles, T, 0, s>>>(L);
  }
  g_result<R><<<blocks_for(L.n_halos, 128), 128, 0, s>>>(L);
  if (L.rows.prof) {
    if (sizeof(R) == 4) g_rows_mixed<<<L.n_halos, T, 0, s>>>(L);
    else g_rows_f64<<<L.n_halos, T, 0, s>>>(L);
  }
  return cudaGetLastError();
}

template <typename R>
int iter_grid_t(int device) {
  int sms = 0, per = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, g_pass<R, true, false, (sizeof(R) == 4 ? 2 : 1)>, T, 0) != cudaSuccess) return 0;
  return sms * (per > 0 ? per : 1);
}

}  // namespace

int grid_iter_grid(int device, int fp64) { return fp64 ? iter_grid_t<double>(device) : iter_grid_t<float>(device); }

int grid_tma_grid(int device) {
  int sms = 0, per = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return 0;
  if (cudaFuncSetAttribute(g_pass_tma, cudaFuncAttributeMaxDynamicSharedMemorySize, TMA_SMEM) != cudaSuccess) return 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, g_pass_tma, T, TMA_SMEM) != cudaSuccess) return 0;
  return sms * per;
}

// The stream (w, r) of n_rows 8-element rows as a 2-D float tensor of 32
// columns, copied in boxes of 32 x 32 (4 KB) with the 128-byte swizzle.
bool grid_wr_map(GridLaunch& L, long long n_rows) {
  using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static Encode encode = nullptr;
  static bool looked = false;
  if (!looked) {
    looked = true;
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      encode = (Encode)fn;
    cudaGetLastError();
  }
  if (!encode || n_rows <= 0 || ((uintptr_t)L.wr & 15)) return false;
  const cuuint64_t dims[2] = {32, (cuuint64_t)n_rows};
  const cuuint64_t strides[1] = {128};
  const cuuint32_t box[2] = {32, 32};
  const cuuint32_t estr[2] = {1, 1};
  return encode(&L.wr_map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, L.wr, dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

cudaError_t grid_bins(GridLaunch& L, cudaStream_t s) { return L.fp64 ? bins_t<double>(L, s) : bins_t<float>(L, s); }

cudaError_t grid_prepare(const GridLaunch& L, cudaStream_t s) {
  return L.fp64 ? prepare_t<double>(L, s) : prepare_t<float>(L, s);
}

cudaError_t grid_sort(GridLaunch& L, cudaStream_t s, unsigned long long or_bits, unsigned long long and_bits) {
  return L.fp64 ? sort_t<double>(L, s, or_bits, and_bits) : sort_t<float>(L, s, or_bits, and_bits);
}

cudaError_t grid_iterate(const GridLaunch& L, int pass, cudaStream_t s) {
  return L.fp64 ? iterate_t<double>(L, pass, s) : iterate_t<float>(L, pass, s);
}

cudaError_t grid_finish(const GridLaunch& L, cudaStream_t s) {
  return L.fp64 ? finish_t<double>(L, s) : finish_t<float>(L, s);
}

}  // namespace ahf
