// Integral properties of bound sets (Sect. 3.1: the spin parameter
// lambda = J sqrt|E| / (G M^(5/2)); the rotation curve's peak) and the
// cross-identification of two catalogues by xi = N_shared^2 / (N_1 N_2)
// (Sect. 3.2).
//
// Properties.  A halo's material within r_vir is its bound list up to k_vir
// (the whole list without an r_vir), in radial order.  The bound lists are
// cut into fixed chunks, one CTA each.  The moments
//   S_m, S_mv, S_md, S_m(d x v), S_m|w|^2, S_mw (w = v + H d), S_m phi
// are accumulated in FP64; with v_bar = S_mv / M they give
// J = S_m(d x v) - S_md x v_bar and
// K = (S_m|w|^2 - 2 v_bar . S_mw + M |v_bar|^2) / 2 = sum m |w - v_bar|^2 / 2.
// The rotation curve's peak is the largest M(<= r_i)^2 / r_i^2 (no square root
// per particle): found in float first, and the particles within 1e-5 of the
// chunk's largest (float is off by 1e-6 at most) settled in FP64.  A final
// kernel adds each halo's chunks in chunk order.
//
// FP64 is what bounds this: the pipe does 1.6 operations a clock and SM.  With
// one mass for all, M(<= r_i) is the particle's place in the list times it and
// one kernel does both parts in 22 FP64 operations a particle (floats become
// doubles on the integer pipes); with a mass each, a second kernel scans the
// masses.  1.2e6 particles of 1,500 haloes: 203 + 233 us
// -> 160 us (kernels alone, caches cold).
//
// Matching.  Every id of the second catalogue is labelled with its halo; one
// CTA per halo of the first catalogue counts the labels of its ids in a
// shared-memory hash table and keeps the largest xi.
#include <algorithm>
#include <cstdint>

#include "ahf_device.cuh"

namespace ahf {
namespace {

constexpr int PT = 256;
constexpr int PER_T = PROPS_CHUNK / PT;   // elements per thread

__device__ __forceinline__ double block_sum_d(double x, double* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  x = warp_sum(x);
  __syncthreads();
  if (lane == 0) red[warp] = x;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < PT / 32; ++w) t += red[w];     // fixed order
  return t;                                            // valid in thread 0
}

__device__ __forceinline__ double to_double(float x) { return float_to_double(x); }
__device__ __forceinline__ double to_double(double x) { return x; }

// Sums over the CTA of NV <= 16 values per thread; value k in thread k.  The
// warps halve the values as they halve the lanes (16 adds a lane in place of 5
// per value), then the warps' sums are added in warp order.
template <int NV>
__device__ __forceinline__ double block_sums(const double s[NV], double* red /* [PT / 32][16] */) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double a[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) a[k] = k < NV ? s[k] : 0.0;
#pragma unroll
  for (int h = 8; h >= 1; h >>= 1) {
    // lanes with bit 2 h keep the upper half of the values
    const bool up = (lane & (2 * h)) != 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (k < h) {
        const double keep = up ? a[k + h] : a[k], give = up ? a[k] : a[k + h];
        a[k] = keep + __shfl_xor_sync(FULL_MASK, give, 2 * h);
      }
    }
  }
  a[0] += __shfl_xor_sync(FULL_MASK, a[0], 1);
  __syncthreads();                       // red may still be read
  // the value a lane ends with: bits 1..4 of the lane, each having picked a half
  if ((lane & 1) == 0) red[warp * 16 + (lane >> 1)] = a[0];
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < NV)
    for (int w = 0; w < PT / 32; ++w) t += red[w * 16 + threadIdx.x];
  return t;
}

// Whether this thread holds the peak: each brings the first of its largest
// M^2 / r^2 at place k of the list (k < 0: none), as cross products find it in list
// order.  Between threads the quotients decide, rounded once each, on ties the
// first in the list, which is the same however the threads are taken; cross products
// M'^2 r^2 > M^2 r'^2 do not order a set where thousands tie to rounding (a flat
// curve), and with the candidates as they arrived the peak differed between calls.
// (A quotient for every particle instead: 20,000 haloes of 40 with a mass each
// 1.4 -> 2.2 ms.)  Thread 0's none when there is no candidate; a NaN mass makes none.
__device__ __forceinline__ bool block_peak(double m, double r2, long long k) {
  __shared__ unsigned long long sq[PT / 32];
  __shared__ long long sk[PT / 32];
  const int n = __syncthreads_count(k >= 0);
  if (n <= 1) return n ? k >= 0 : threadIdx.x == 0;      // mostly one thread's
  unsigned long long best = 0;           // the quotient's bits, which order as it does
  long long at = k;
  auto take = [&](unsigned long long q, long long k2) {
    const bool before = k2 >= 0 && (at < 0 || q > best || (q == best && k2 < at));
    best = before ? q : best;
    at = before ? k2 : at;
  };
  if (__any_sync(FULL_MASK, k >= 0)) {
    const double q = k >= 0 ? m * m / r2 : 0.0;
    if (q >= 0.0) best = (unsigned long long)__double_as_longlong(q);
    else at = -1;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long q2 = __shfl_xor_sync(FULL_MASK, best, o);
      const long long k2 = __shfl_xor_sync(FULL_MASK, at, o);
      take(q2, k2);
    }
  }
  if ((threadIdx.x & 31) == 0) {
    sq[threadIdx.x >> 5] = best;
    sk[threadIdx.x >> 5] = at;
  }
  __syncthreads();
#pragma unroll
  for (int w = 0; w < PT / 32; ++w) take(sq[w], sk[w]);
  return at < 0 ? threadIdx.x == 0 : at == k;
}

// The largest of one float >= 0 per thread over the CTA.
__device__ __forceinline__ float block_max(float x, uint32_t* word) {
  if (threadIdx.x == 0) *word = 0u;
  __syncthreads();
  const uint32_t w = __reduce_max_sync(FULL_MASK, __float_as_uint(x));
  if ((threadIdx.x & 31) == 0) atomicMax(word, w);
  __syncthreads();
  return __uint_as_float(*word);
}

// x > 0, neither subnormal nor infinite nor NaN
__device__ __forceinline__ bool is_normal(float x) { return __float_as_uint(x) - 0x800000u < 0x7f000000u; }

// The float M^2 / r^2 a particle is first judged by: within 1e-6 of the exact
// value while M^2, r^2 and their quotient are normal floats; where one is not
// (SI units: r^2 ~ 1e42; masses below 1e-19), infinite, which leaves the chunk to
// FP64.  -1: at the centre (r2 = 0).
__device__ __forceinline__ float peak_guess(float m, float r2f, double r2) {
  const float m2 = m * m, q = m2 / r2f;
  if (is_normal(m2) && is_normal(r2f) && is_normal(q)) return q;
  return r2 > 0.0 ? INFINITY : -1.0f;
}
// What it has to reach: the chunk's largest less 1e-5 (all of them when float
// cannot hold it).
__device__ __forceinline__ float peak_least(float largest) {
  return isfinite(largest) ? largest * (1.0f - 1e-5f) : 0.0f;
}

// Offset from the centre in FP64 (minimum image in a periodic box), velocity
// and mass of particle pi.
template <int CT>
__device__ __forceinline__ void load_f64(const PropsLaunch& L, const HaloDev& H, long long pi, double d[3], double v[3],
                                         double& m) {
  Cand<CT> c;
  load_cand<CT>(L.p, pi, c);
  const double x[3] = {to_double(c.x), to_double(c.y), to_double(c.z)};
  const double box = L.frame.box;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    double t = x[a] - H.c[a];
    if (box > 0.0) {
      const double half = 0.5 * box;
      if (t > half) t -= box;
      else if (t < -half) t += box;
    }
    d[a] = t;
  }
  v[0] = to_double(c.vx);
  v[1] = to_double(c.vy);
  v[2] = to_double(c.vz);
  m = L.p.m ? to_double(c.m) : L.p.m0;
}

__device__ __forceinline__ long long n_used(const ahf_result& r) {
  return r.k_vir >= 0 ? r.k_vir + 1 : r.n_bound;
}

__device__ __forceinline__ double load_phi(const PropsLaunch& L, long long slot) {
  return L.phi_f64 ? ((const double*)L.phi)[slot] : float_to_double(((const float*)L.phi)[slot]);
}

// One mass for all: the moments and the peak of one chunk.
template <int CT>
__global__ void __launch_bounds__(PT) props_uniform(PropsLaunch L) {
  __shared__ double red[PT / 32 * 16];
  __shared__ uint32_t word;
  const int c = blockIdx.x;
  const int h = L.chunk_halo[c];
  const HaloDev& H = L.halos[h];
  const long long n = n_used(L.res[h]);
  const long long start = L.chunk_start[c];
  const int ne = (int)max(0ll, min(n - start, (long long)PROPS_CHUNK));
  double* out = L.part + (size_t)c * PROPS_PART;
  if (ne == 0) {
    if (threadIdx.x == 0) out[15] = 0.0;
    return;
  }
  const long long* list = L.bound_idx + H.offset + start;
  // v, d, d x v, |w|^2, phi
  double s[11];
#pragma unroll
  for (int k = 0; k < 11; ++k) s[k] = 0.0;
  float q[PER_T], qm = 0.0f;
#pragma unroll
  for (int j0 = 0; j0 < PER_T; j0 += 2) {
    if (j0 * PT >= ne) break;
#pragma unroll
    for (int j = j0; j < j0 + 2; ++j) {
      const int e = j * PT + threadIdx.x;
      q[j] = -1.0f;
      if (e >= ne) continue;
      double d[3], v[3], m;
      load_f64<CT>(L, H, list[e], d, v, m);
      const double phi = load_phi(L, H.offset + start + e);
      double w2 = s[9];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        s[a] += v[a];
        s[3 + a] += d[a];
        const double w = fma(L.H, d[a], v[a]);
        w2 = fma(w, w, w2);
      }
      s[9] = w2;
      s[6] = fma(d[1], v[2], fma(-d[2], v[1], s[6]));
      s[7] = fma(d[2], v[0], fma(-d[0], v[2], s[7]));
      s[8] = fma(d[0], v[1], fma(-d[1], v[0], s[8]));
      s[10] += phi;
      const float fx = double_to_float(d[0]), fy = double_to_float(d[1]), fz = double_to_float(d[2]);
      const float r2f = fmaf(fz, fz, fmaf(fy, fy, fx * fx));
      q[j] = peak_guess((float)(int)(start + e + 1), r2f,
                        is_normal(r2f) ? 1.0 : d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
      qm = fmaxf(qm, q[j]);
    }
  }
  const double t = block_sums<11>(s, red);
  if (threadIdx.x < 11) red[threadIdx.x] = t * L.p.m0;
  const float least = peak_least(block_max(qm, &word));      // (its barriers order red)
  if (threadIdx.x == 0) {
    out[0] = (double)ne * L.p.m0;
    for (int a = 0; a < 3; ++a) {
      out[1 + a] = red[a];
      out[4 + a] = red[3 + a];
      out[7 + a] = red[6 + a];
      out[11 + a] = fma(L.H, red[3 + a], red[a]);
    }
    out[10] = red[9];
    out[14] = red[10];
    out[15] = (double)ne;
  }
  double bm = 0.0, br = 0.0;
  long long bk = -1;
#pragma unroll
  for (int j = 0; j < PER_T; ++j) {
    if (j * PT >= ne) break;
    if (q[j] < least || q[j] < 0.0f) continue;
    const int e = j * PT + threadIdx.x;
    double d[3], v[3], m;
    load_f64<CT>(L, H, list[e], d, v, m);
    const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    const double cum = (double)(start + e + 1);
    if (r2 > 0.0 && (bk < 0 || cum * cum * br > bm * bm * r2)) {
      bm = cum;
      br = r2;
      bk = start + e;
    }
  }
  if (block_peak(bm, br, bk)) {
    out[16] = bm * L.p.m0;
    out[17] = br;
    out[18] = (double)bk;
  }
}

// A mass each: the moments of one chunk.
template <int CT>
__global__ void __launch_bounds__(PT) props_moments(PropsLaunch L) {
  __shared__ double red[PT / 32 * 16];
  const int c = blockIdx.x;
  const int h = L.chunk_halo[c];
  const HaloDev& H = L.halos[h];
  const long long n = n_used(L.res[h]);
  const long long start = L.chunk_start[c];
  const long long end = min(n, start + (long long)PROPS_CHUNK);
  double s[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) s[k] = 0.0;
  for (long long k = start + threadIdx.x; k < end; k += PT) {
    const long long pi = L.bound_idx[H.offset + k];
    double d[3], v[3], m;
    load_f64<CT>(L, H, pi, d, v, m);
    const double phi = load_phi(L, H.offset + k);
    double w2 = 0.0;
    s[0] += m;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const double w = fma(L.H, d[a], v[a]);
      w2 = fma(w, w, w2);
      s[1 + a] = fma(m, v[a], s[1 + a]);
      s[4 + a] = fma(m, d[a], s[4 + a]);
    }
    s[7] = fma(m, d[1] * v[2] - d[2] * v[1], s[7]);
    s[8] = fma(m, d[2] * v[0] - d[0] * v[2], s[8]);
    s[9] = fma(m, d[0] * v[1] - d[1] * v[0], s[9]);
    s[10] = fma(m, w2, s[10]);
    s[11] = fma(m, phi, s[11]);
  }
  double* out = L.part + (size_t)c * PROPS_PART;
  const double t = block_sums<12>(s, red);
  if (threadIdx.x < 11) out[threadIdx.x] = t;
  if (threadIdx.x == 11) out[14] = t;
  __syncthreads();
  if (threadIdx.x < 12) red[threadIdx.x] = t;
  __syncthreads();
  if (threadIdx.x < 3) out[11 + threadIdx.x] = fma(L.H, red[4 + threadIdx.x], red[1 + threadIdx.x]);
  if (threadIdx.x == 0) out[15] = (double)max(0ll, end - start);
}

// A mass each: the rotation curve's peak within one chunk, M(<= r_i) from the
// chunk's offset (the earlier chunks' masses) and a block scan.
template <int CT>
__global__ void __launch_bounds__(PT) props_vmax(PropsLaunch L) {
  __shared__ double red[PT / 32];
  __shared__ double wtot[PT / 32];
  __shared__ double m_off;
  __shared__ uint32_t word;
  const int c = blockIdx.x;
  const int h = L.chunk_halo[c];
  const HaloDev& H = L.halos[h];
  const long long n = n_used(L.res[h]);
  const long long start = L.chunk_start[c];
  const long long end = min(n, start + (long long)PROPS_CHUNK);
  if (start >= end) return;              // its part counts for nothing
  // the mass of the halo's earlier chunks, added in chunk order
  double pre = 0.0;
  for (int k = L.halo_chunk0[h] + (int)threadIdx.x; k < c; k += PT) pre += L.part[(size_t)k * PROPS_PART];
  const double off = block_sum_d(pre, red);
  if (threadIdx.x == 0) m_off = off;
  // this thread's run of consecutive elements: masses and squared radii
  const long long k0 = start + (long long)threadIdx.x * PER_T;
  double m[PER_T], r2[PER_T];
  double run = 0.0;
#pragma unroll
  for (int j = 0; j < PER_T; ++j) {
    m[j] = 0.0;
    r2[j] = 0.0;
    const long long k = k0 + j;
    if (k < end) {
      double d[3], v[3];
      load_f64<CT>(L, H, L.bound_idx[H.offset + k], d, v, m[j]);
      r2[j] = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    }
    run += m[j];
  }
  // exclusive block scan of the runs' masses
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double inc = run;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double y = __shfl_up_sync(FULL_MASK, inc, o);
    if (lane >= o) inc += y;
  }
  __syncthreads();
  if (lane == 31) wtot[warp] = inc;
  __syncthreads();
  double base = m_off;
  for (int w = 0; w < warp; ++w) base += wtot[w];
  base += inc - run;
  float q[PER_T], qm = 0.0f;
  double cum = base;
#pragma unroll
  for (int j = 0; j < PER_T; ++j) {
    cum += m[j];
    m[j] = cum;                          // the inclusive mass from here on
    q[j] = k0 + j < end ? peak_guess(double_to_float(cum), double_to_float(r2[j]), r2[j]) : -1.0f;
    qm = fmaxf(qm, q[j]);
  }
  const float least = peak_least(block_max(qm, &word));
  // the largest M(<= r_i) / r_i of the run (first one on ties)
  double best_m = 0.0, best_r2 = 0.0;
  long long best_k = -1;
#pragma unroll
  for (int j = 0; j < PER_T; ++j) {
    if (q[j] < least || q[j] < 0.0f) continue;
    if (r2[j] > 0.0 && (best_k < 0 || m[j] * m[j] * best_r2 > best_m * best_m * r2[j])) {
      best_m = m[j];
      best_r2 = r2[j];
      best_k = k0 + j;
    }
  }
  if (block_peak(best_m, best_r2, best_k)) {
    double* out = L.part + (size_t)c * PROPS_PART;
    out[16] = best_m;
    out[17] = best_r2;
    out[18] = (double)best_k;
  }
}

// One thread per halo: add the chunks in order and form the properties.
__global__ void props_final(PropsLaunch L) {
  const int h = blockIdx.x * blockDim.x + threadIdx.x;
  if (h >= L.n_halos) return;
  const ahf_result r = L.res[h];
  const long long n = n_used(r);
  double* o = L.props + (size_t)h * AHF_PROP_FIELDS;
  for (int k = 0; k < AHF_PROP_FIELDS; ++k) o[k] = 0.0;
  o[11] = r.k_vir >= 0 ? 1.0 : 0.0;
  if (n <= 0) return;
  double s[15];
  for (int k = 0; k < 15; ++k) s[k] = 0.0;
  double mb = 0.0, rb = 0.0, kb = -1.0;
  for (int c = L.halo_chunk0[h]; c < L.halo_chunk0[h + 1]; ++c) {
    const double* p = L.part + (size_t)c * PROPS_PART;
    if (p[15] <= 0.0) continue;
    for (int k = 0; k < 15; ++k) s[k] += p[k];
    if (p[18] >= 0.0 && (kb < 0.0 || p[16] * p[16] * rb > mb * mb * p[17])) {
      mb = p[16];
      rb = p[17];
      kb = p[18];
    }
  }
  const double M = s[0];
  const double vb[3] = {s[1] / M, s[2] / M, s[3] / M};
  const double J[3] = {s[7] - (s[5] * vb[2] - s[6] * vb[1]), s[8] - (s[6] * vb[0] - s[4] * vb[2]),
                       s[9] - (s[4] * vb[1] - s[5] * vb[0])};
  const double K = 0.5 * (s[10] - 2.0 * (vb[0] * s[11] + vb[1] * s[12] + vb[2] * s[13]) +
                          M * (vb[0] * vb[0] + vb[1] * vb[1] + vb[2] * vb[2]));
  const double U = 0.5 * s[14];
  const double E = K + U;
  const double Jn = sqrt(J[0] * J[0] + J[1] * J[1] + J[2] * J[2]);
  o[0] = (double)n;
  o[1] = M;
  o[2] = J[0];
  o[3] = J[1];
  o[4] = J[2];
  o[5] = K;
  o[6] = U;
  o[7] = E;
  o[8] = Jn * sqrt(fabs(E)) / (L.G * M * M * sqrt(M));
  if (kb >= 0.0) {
    const double rmax = sqrt(rb);
    o[9] = sqrt(L.G * mb / rmax);
    o[10] = rmax;
  }
}

// ---- matching ----------------------------------------------------------------

constexpr int M_UNROLL = 4;              // ids in flight per thread

// The ids of halo blockIdx.x, spread over gridDim.y CTAs.
__global__ void __launch_bounds__(PT) match_label(MatchLaunch L) {
  const int b = blockIdx.x;
  const long long off = L.off_b[b], cnt = L.cnt_b[b];
  const long long step = (long long)gridDim.y * PT;
  for (long long k0 = (long long)blockIdx.y * PT + threadIdx.x; k0 < cnt; k0 += M_UNROLL * step) {
    long long id[M_UNROLL];
    int old[M_UNROLL];
#pragma unroll
    for (int j = 0; j < M_UNROLL; ++j) id[j] = k0 + j * step < cnt ? L.ids_b[off + k0 + j * step] : 0;
#pragma unroll
    for (int j = 0; j < M_UNROLL; ++j) {
      old[j] = b;
      if (k0 + j * step >= cnt) continue;
      if (id[j] < 0 || id[j] >= L.n_ids) atomicOr(L.err, ERR_ID_RANGE);
      else old[j] = atomicCAS(&L.label[id[j]], -1, b);
    }
#pragma unroll
    for (int j = 0; j < M_UNROLL; ++j)
      if (old[j] != -1 && old[j] != b) atomicOr(L.err, ERR_SHARED_ID);
  }
}

// One CTA per halo: its ids' labels counted in a hash table, a thread adding
// only when the label changes (a halo's particles mostly share one: an add per
// id queued on one counter, and one thread's search of the table cost as much;
// 182 -> 53 us for 1,500 haloes of 1.2e6 ids, caches cold).
constexpr int MT = 512;

__global__ void __launch_bounds__(MT) match_best(MatchLaunch L) {
  __shared__ int key[MATCH_TABLE];
  __shared__ int cnt[MATCH_TABLE];
  __shared__ int overflow;
  __shared__ double bx[MT / 32];
  __shared__ int bb[MT / 32], bc[MT / 32];
  const int a = blockIdx.x;
  for (int i = threadIdx.x; i < MATCH_TABLE; i += MT) {
    key[i] = -1;
    cnt[i] = 0;
  }
  if (threadIdx.x == 0) overflow = 0;
  __syncthreads();
  const long long off = L.off_a[a], na = L.cnt_a[a];
  auto add = [&](int b, int n) {
    unsigned slot = ((unsigned)b * 2654435761u) & (MATCH_TABLE - 1);
    for (int probe = 0; probe < MATCH_TABLE; ++probe) {   // bounded: at most every slot once
      const int k0 = atomicCAS(&key[slot], -1, b);
      if (k0 == -1 || k0 == b) {
        atomicAdd(&cnt[slot], n);
        return;
      }
      slot = (slot + 1) & (MATCH_TABLE - 1);
    }
    overflow = 1;
  };
  int cur = -1, run = 0;
  for (long long k0 = threadIdx.x; k0 < na; k0 += (long long)M_UNROLL * MT) {
    long long id[M_UNROLL];
    int lab[M_UNROLL];
#pragma unroll
    for (int j = 0; j < M_UNROLL; ++j) {
      const long long k = k0 + (long long)j * MT;
      id[j] = k < na ? L.ids_a[off + k] : 0;
    }
#pragma unroll
    for (int j = 0; j < M_UNROLL; ++j) {
      lab[j] = -1;
      if (k0 + (long long)j * MT >= na) continue;
      if (id[j] < 0 || id[j] >= L.n_ids) atomicOr(L.err, ERR_ID_RANGE);
      else lab[j] = L.label[id[j]];
    }
#pragma unroll
    for (int j = 0; j < M_UNROLL; ++j) {
      if (lab[j] < 0) continue;
      if (lab[j] != cur) {
        if (run) add(cur, run);
        cur = lab[j];
        run = 0;
      }
      ++run;
    }
  }
  if (run) add(cur, run);
  __syncthreads();
  // the largest xi, the lower halo on ties
  double x = 0.0;
  int b = -1, c = 0;
  auto take = [&](double x2, int b2, int c2) {
    if (b2 >= 0 && (b < 0 || x2 > x || (x2 == x && b2 < b))) {
      x = x2;
      b = b2;
      c = c2;
    }
  };
  for (int i = threadIdx.x; i < MATCH_TABLE; i += MT) {
    const int b2 = key[i];
    if (b2 < 0) continue;
    const double n = (double)cnt[i];
    take(n * n / ((double)na * (double)L.cnt_b[b2]), b2, cnt[i]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double x2 = __shfl_xor_sync(FULL_MASK, x, o);
    const int b2 = __shfl_xor_sync(FULL_MASK, b, o), c2 = __shfl_xor_sync(FULL_MASK, c, o);
    take(x2, b2, c2);
  }
  if ((threadIdx.x & 31) == 0) {
    bx[threadIdx.x >> 5] = x;
    bb[threadIdx.x >> 5] = b;
    bc[threadIdx.x >> 5] = c;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < MT / 32; ++w) take(bx[w], bb[w], bc[w]);
    if (overflow) {
      atomicOr(L.err, ERR_MATCH_TABLE);
      b = -2;
      x = 0.0;
      c = 0;
    }
    L.best[a] = b;
    L.shared[a] = c;
    L.xi[a] = b >= 0 ? x : 0.0;
  }
}

}  // namespace

cudaError_t launch_properties(const PropsLaunch& L, cudaStream_t s) {
  if (L.n_halos == 0) return cudaSuccess;
  const bool f64 = L.p.coord_type == AHF_COORD_F64;
  if (L.n_chunks > 0 && L.p.m == nullptr) {
    if (f64) props_uniform<AHF_COORD_F64><<<L.n_chunks, PT, 0, s>>>(L);
    else props_uniform<AHF_COORD_F32_REL><<<L.n_chunks, PT, 0, s>>>(L);
  } else if (L.n_chunks > 0) {
    if (f64) {
      props_moments<AHF_COORD_F64><<<L.n_chunks, PT, 0, s>>>(L);
      props_vmax<AHF_COORD_F64><<<L.n_chunks, PT, 0, s>>>(L);
    } else {
      props_moments<AHF_COORD_F32_REL><<<L.n_chunks, PT, 0, s>>>(L);
      props_vmax<AHF_COORD_F32_REL><<<L.n_chunks, PT, 0, s>>>(L);
    }
  }
  props_final<<<(L.n_halos + 31) / 32, 32, 0, s>>>(L);   // FP64 latency: spread over the SMs
  return cudaGetLastError();
}

cudaError_t launch_match(const MatchLaunch& L, cudaStream_t s) {
  // The list lengths are on the device.  One CTA took 130 us over a halo of 41,000
  // ids, so a halo gets up to 64 (of 4 ids a thread) while that is 64 an SM in all
  // at most.  (Four times as many, of an id a thread, took as long over long lists
  // but had mostly nothing to do for short ones: 600 haloes of 100 ids, a call
  // alone, 63 us; one CTA a halo 55; now 50.)
  if (L.n_b > 0) {
    const int shares = std::min(64, std::max(1, 64 * L.sms / L.n_b));
    match_label<<<dim3((unsigned)L.n_b, (unsigned)shares), PT, 0, s>>>(L);
  }
  if (L.n_a > 0) match_best<<<L.n_a, MT, 0, s>>>(L);
  return cudaGetLastError();
}

}  // namespace ahf
