// On-chip classes: a halo unbound entirely in shared memory, by one CTA or
// by a thread-block cluster of CS CTAs sharing their shared memory (DSMEM).
//
// Per halo (Sect. 2.1 and Appendix A):
//   gather   candidates -> (radius key, candidate position), FP64-accurate
//            recentring and sphere test, exponent maxima for the exact sums;
//            each member's offset, mass and velocity to its 32-byte record
//   sort     by radius, stable, once: the centre is fixed and
//            particles only leave, so the survivors of every later iteration
//            stay in radial order.  One CTA distributes (dist_sort; count_sort
//            for dozens of equal radii); a cluster first hands every CTA its
//            share of the order (cluster_dist_sort; cluster_radix_sort when a
//            share would not fit).
//   fill     sorted SoA from the records: radius, mass, w = v + H d; exact
//            sum m v
//   iterate  scan of the exact M(<r) and sum m/r prefixes ->
//            phi_i = -G [M(<r_i)/r_i + sum_{j>=i} m_j/r_j], escape test
//            |w - v_bulk|^2 > 2|phi|, removal of every unbound particle, until
//            an iteration removes nothing.  Each thread keeps the exact sums
//            of its own particles and subtracts what it removes, so one pass
//            over the particles per iteration suffices.
//   emit     bound list (particle index, phi) in radial order, virial crossing
//            of the final set (Sect. 2.1, Eqs. 1-2), result record
//
// CTAs (clusters) are persistent: each pulls the next halo from a counter over
// the class's haloes, which the host orders largest first.  Cross-CTA values
// go through a small exchange record in each CTA's shared memory, read by the
// others after a hardware cluster barrier; every CTA combines them in rank
// order, so all CTAs hold identical cluster-wide values.
#include <cooperative_groups.h>

#include <cstdint>

#include "ahf_device.cuh"

namespace cg = cooperative_groups;

namespace ahf {
namespace {

template <int CS>
struct Cl {
  static __device__ __forceinline__ int rank() {
    if constexpr (CS > 1) return (int)cg::this_cluster().block_rank();
    else return 0;
  }
  static __device__ __forceinline__ void sync() {
    if constexpr (CS > 1) cg::this_cluster().sync();
    else __syncthreads();
  }
  template <typename T>
  static __device__ __forceinline__ T* at(T* p, int r) {
    if constexpr (CS > 1) return cg::this_cluster().map_shared_rank(p, r);
    else return p;
  }
};

// Largest bin count a cluster forms profile rows for itself (larger requests
// use the profile kernels).
constexpr int FUSE_BINS = 128;

// Values a CTA publishes to the other CTAs of its cluster.
struct Xchg {
  int halo;
  uint32_t g_or, g_and, g_mxm, g_mxr, g_mxv, g_kmx, g_kmn;
  int g_nmem;
  uint32_t cnt[256];            // radix pass: digit counts of this CTA; dist sort: its
                                // members bound for each CTA
  long long mv[3];              // fill: partial sum m v
  // iteration exchange, two alternating copies: scan totals of this CTA
  // (M, sum m/r, count) and its removals of the previous iteration (m,
  // m v (3), count, band count)
  long long xt[2][3];
  long long xr[2][4];
  int xn[2], xb[2];
  float first_r;                // emit: first compacted radius of this CTA
  int nb_loc;                   // emit: bound particles held by this CTA
  int kf;                       // emit: first local virial crossing (global index)
  // fused profile rows: r_vir and the outermost radius, from the CTAs that hold
  // them; the bound count at every bin edge (all CTAs', in rank 0) and this CTA's
  // inclusive mass there
  double rvir;
  float last_r;
  int pc[FUSE_BINS + 1];
  long long pm[FUSE_BINS + 1];
};

template <int NT>
struct Smem {
  static constexpr int NW = NT / 32;
  long long red[NW][4];
  long long scan_base[NW][3];
  long long tot[3];
  uint32_t or_bits, and_bits, max_m, max_mr, max_mv;
  uint32_t max_key, min_key;    // extreme member keys
  int n_member;
  long long acc[4];             // block accumulators (m v or removed m, m v)
  int acc_n, acc_band;
  // one CTA's removal sums, alternating between iterations: (removed m, m v),
  // removed count, band count
  long long racc[2][4];
  int racc_n[2], racc_band[2];
  // cluster-wide values
  long long c_pre[3];           // exclusive prefix over lower ranks
  long long c_tot[3];
  long long mv[3];              // exact sum m v of the current set
  int c_removed, c_band;
  int k_first;
  float vb[3];
  double rvir;                  // emit: the record's r_vir and k_vir, for the profile rows
  long long kvir;
  uint32_t dtot[256];
  uint32_t dpre[256];
};

template <int NT>
__device__ __forceinline__ void block_exclusive_scan3(long long& a, long long& b, long long& c, Smem<NT>& S) {
  constexpr int NW = NT / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  long long ia = warp_inclusive_scan(a, lane);
  long long ib = warp_inclusive_scan(b, lane);
  long long ic = warp_inclusive_scan(c, lane);
  if (lane == 31) { S.red[warp][0] = ia; S.red[warp][1] = ib; S.red[warp][2] = ic; }
  __syncthreads();
  if (warp == 0) {
    long long x = lane < NW ? S.red[lane][0] : 0, y = lane < NW ? S.red[lane][1] : 0,
              z = lane < NW ? S.red[lane][2] : 0;
    long long sx = warp_inclusive_scan(x, lane), sy = warp_inclusive_scan(y, lane), sz = warp_inclusive_scan(z, lane);
    if (lane < NW) { S.scan_base[lane][0] = sx - x; S.scan_base[lane][1] = sy - y; S.scan_base[lane][2] = sz - z; }
    if (lane == NW - 1) { S.tot[0] = sx; S.tot[1] = sy; S.tot[2] = sz; }
  }
  __syncthreads();
  a = S.scan_base[warp][0] + ia - a;
  b = S.scan_base[warp][1] + ib - b;
  c = S.scan_base[warp][2] + ic - c;
}

// The same for two values (the iterations need no count): totals in
// S.tot[0], S.tot[1].
template <int NT>
__device__ __forceinline__ void block_exclusive_scan2(long long& a, long long& b, Smem<NT>& S) {
  constexpr int NW = NT / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  long long ia = warp_inclusive_scan(a, lane);
  long long ib = warp_inclusive_scan(b, lane);
  if (lane == 31) { S.red[warp][0] = ia; S.red[warp][1] = ib; }
  __syncthreads();
  if (warp == 0) {
    long long x = lane < NW ? S.red[lane][0] : 0, y = lane < NW ? S.red[lane][1] : 0;
    long long sx = warp_inclusive_scan(x, lane), sy = warp_inclusive_scan(y, lane);
    if (lane < NW) { S.scan_base[lane][0] = sx - x; S.scan_base[lane][1] = sy - y; }
    if (lane == NW - 1) { S.tot[0] = sx; S.tot[1] = sy; }
  }
  __syncthreads();
  a = S.scan_base[warp][0] + ia - a;
  b = S.scan_base[warp][1] + ib - b;
}

// One exchange of a cluster iteration: every CTA publishes its scan totals
// of the current set and its removal sums of the previous iteration (zero
// before the first) in copy `xs`, and combines the cluster's: S.c_pre gets
// the totals over lower ranks, S.c_tot over all ranks; S.mv loses the m v
// removed, S.c_removed and S.c_band count the removed and the band.  The
// copies alternate between iterations: a CTA writes copy xs again only
// after the next exchange's barrier, which every reader of this one has
// passed after reading it.
template <int NT, int CS>
__device__ __forceinline__ void cluster_exchange(Smem<NT>& S, Xchg& X, int rank, int xs, bool first) {
  if (threadIdx.x == 0) {
    X.xt[xs][0] = S.tot[0]; X.xt[xs][1] = S.tot[1]; X.xt[xs][2] = S.tot[2];
    X.xr[xs][0] = first ? 0 : S.acc[0];
    X.xr[xs][1] = first ? 0 : S.acc[1];
    X.xr[xs][2] = first ? 0 : S.acc[2];
    X.xr[xs][3] = first ? 0 : S.acc[3];
    X.xn[xs] = first ? 0 : S.acc_n;
    X.xb[xs] = first ? 0 : S.acc_band;
  }
  Cl<CS>::sync();
  if (threadIdx.x < 3) {
    long long pre = 0, tot = 0;
#pragma unroll
    for (int r = 0; r < CS; ++r) {
      const long long v = Cl<CS>::at(&X.xt[xs][0], r)[threadIdx.x];
      if (r < rank) pre += v;
      tot += v;
    }
    S.c_pre[threadIdx.x] = pre;
    S.c_tot[threadIdx.x] = tot;
  } else if (threadIdx.x == 32) {
    long long a1 = 0, a2 = 0, a3 = 0;
    int nr = 0, nbd = 0;
#pragma unroll
    for (int r = 0; r < CS; ++r) {
      const Xchg* Y = Cl<CS>::at(&X, r);
      a1 += Y->xr[xs][1]; a2 += Y->xr[xs][2]; a3 += Y->xr[xs][3];
      nr += Y->xn[xs]; nbd += Y->xb[xs];
    }
    S.mv[0] -= a1; S.mv[1] -= a2; S.mv[2] -= a3;
    S.c_removed = nr;
    S.c_band = nbd;
  }
  __syncthreads();
}

// Stable LSD radix sort of the halo's keys, 8-bit digits, skipping the digits
// in which all keys agree.  Each CTA of the cluster holds `nloc` elements of a
// chunk of `chunk` positions, in order; the result keeps that partition.  Every pass scatters (key, value) pairs
// as one 8-byte store into the owner CTA's shared memory (the two arrays of a
// buffer, kA|vA or kB|vB, hold CAP interleaved pairs between passes); a local
// pass splits the final pairs into the other buffer.  Returns 0 if the result
// is in (kA, vA), 1 if in (kB, vB) (the same in every CTA).
template <int NT, int IPT, int CS>
__device__ int cluster_radix_sort(uint32_t* kA, uint32_t* vA, uint32_t* kB, uint32_t* vB, uint16_t* hist, Smem<NT>& S,
                                  Xchg& X, int nloc, int chunk, uint32_t diff, int rank) {
  constexpr int NW = NT / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int passes[4], np = 0;
  for (int d = 0; d < 4; ++d)
    if ((diff >> (8 * d)) & 0xffu) passes[np++] = d;
  if (np == 0) {
    for (int p = threadIdx.x; p < nloc; p += NT) {
      kB[p] = kA[p];
      vB[p] = vA[p];
    }
    __syncthreads();
    return 1;
  }
  uint2* pA = reinterpret_cast<uint2*>(kA);     // kA|vA as interleaved pairs
  uint2* pB = reinterpret_cast<uint2*>(kB);     // kB|vB
  uint2 *pin = pA, *pout = pB;
  const int wchunk = ((nloc + NW * 32 - 1) / (NW * 32)) * 32;   // per-warp run
  const int nb = wchunk / 32;                                   // <= IPT
  for (int ip = 0; ip < np; ++ip) {
    const int shift = 8 * passes[ip];
    for (int i = threadIdx.x; i < NW * 256; i += NT) hist[i] = 0;
    __syncthreads();
    // keys are read again for the scatter (the input buffer does not change
    // during a pass): only the ranks stay in registers
    uint16_t rank_in[IPT];
#pragma unroll
    for (int b = 0; b < IPT; ++b) {
      if (b < nb) {
        const int e = warp * wchunk + b * 32 + lane;
        const bool valid = e < nloc;
        const uint32_t key = valid ? (ip == 0 ? kA[e] : pin[e].x) : 0u;   // pass 0: the gather's arrays
        const unsigned vmask = __ballot_sync(FULL_MASK, valid);
        rank_in[b] = 0;
        if (valid) {
          const uint32_t dg = (key >> shift) & 0xffu;
          const unsigned peers = __match_any_sync(vmask, dg);
          const unsigned below = peers & lanemask_lt();
          const uint16_t base = hist[warp * 256 + dg];
          rank_in[b] = (uint16_t)(base + __popc(below));
          __syncwarp(vmask);
          if (below == 0) hist[warp * 256 + dg] = (uint16_t)(base + __popc(peers));
        }
        __syncwarp();
      }
    }
    __syncthreads();
    // this CTA's digit counts; per-warp counts become within-CTA offsets
    for (int dg = threadIdx.x; dg < 256; dg += NT) {
      uint32_t run = 0;
      for (int w = 0; w < NW; ++w) {
        const uint32_t h = hist[w * 256 + dg];
        hist[w * 256 + dg] = (uint16_t)run;
        run += h;
      }
      X.cnt[dg] = run;
    }
    Cl<CS>::sync();
    // cluster: digit totals, and counts of this digit in lower-ranked CTAs
    for (int dg = threadIdx.x; dg < 256; dg += NT) {
      uint32_t tot = 0, pre = 0;
      for (int r = 0; r < CS; ++r) {
        const uint32_t v = Cl<CS>::at(X.cnt, r)[dg];
        if (r < rank) pre += v;
        tot += v;
      }
      S.dtot[dg] = tot;
      S.dpre[dg] = pre;
    }
    __syncthreads();
    if (warp == 0) {
      uint32_t loc[8], s = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) { loc[i] = S.dtot[lane * 8 + i]; s += loc[i]; }
      const uint32_t inc = warp_inclusive_scan(s, lane);
      uint32_t run = inc - s;
#pragma unroll
      for (int i = 0; i < 8; ++i) { S.dtot[lane * 8 + i] = run + S.dpre[lane * 8 + i]; run += loc[i]; }
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < IPT; ++b) {
      if (b < nb) {
        const int e = warp * wchunk + b * 32 + lane;
        if (e < nloc) {
          const uint2 kv = ip == 0 ? make_uint2(kA[e], vA[e]) : pin[e];
          const uint32_t dg = (kv.x >> shift) & 0xffu;
          const int g = (int)S.dtot[dg] + (int)hist[warp * 256 + dg] + (int)rank_in[b];
          const int q = g / chunk;
          Cl<CS>::at(pout, q)[g - q * chunk] = kv;
        }
      }
    }
    Cl<CS>::sync();
    uint2* t = pin;
    pin = pout;
    pout = t;
  }
  // split this CTA's sorted pairs into the other buffer
  uint32_t* ko = reinterpret_cast<uint32_t*>(pout);
  uint32_t* vo = ko + IPT * NT;
  for (int p = threadIdx.x; p < nloc; p += NT) {
    const uint2 x = pin[p];
    ko[p] = x.x;
    vo[p] = x.y;
  }
  __syncthreads();
  return pout == pA ? 0 : 1;
}

constexpr int SORT_CELLS = 512;     // cells of a CTA's radial sort
constexpr int CLUSTER_CELLS = 1024; // cells a cluster divides its members by

// The radial sort of a cluster by distribution: the members are counted in
// cells over the whole halo; the cells' counts give every CTA an equal share of
// the order (within the few members by which a cell is not linear); each member
// goes to the CTA of its share, once; every CTA sorts what it got (dist_sort).
// Four cluster barriers and one DSMEM store per member, where the radix sort
// takes two barriers, a ranking by lane matching and a store per key byte:
// 42 -> 20 us per halo in clusters of 2 and 4 CTAs, 46 -> 23 of 8, 55 -> 23 of 16.
// CTA r's share is radially below CTA r + 1's; what it holds is its own (nrec;
// not the chunk of the candidates), in order, in (kA, vA) of every CTA (0
// returned).  -1, with everything as it was, when a share would not fit.
template <int NT, int IPT, int CS>
__device__ int cluster_dist_sort(uint32_t* kA, uint32_t* vA, uint32_t* kB, uint32_t* vB, uint32_t* ex1, uint32_t* ex2,
                                 uint32_t* hist, Smem<NT>& S, Xchg& X, int nloc, int n_mem, int rank, int& nrec) {
  constexpr int NW = NT / 32, CAP = IPT * NT, SLICE = CLUSTER_CELLS / CS;
  static_assert(SLICE <= NT && CLUSTER_CELLS % NT == 0 && NW * 16 <= NT,
                "slices and counters fit the threads");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t* mine = ex2;                  // this CTA's cells
  uint32_t* cum = ex1;                   // all of them: counts, then members before each cell
  uint32_t* wq = hist;                   // [NW][16] members of each warp per destination
  uint32_t* wtot = reinterpret_cast<uint32_t*>(&S.red[0][0]);
  const uint32_t kmin = S.min_key, range = S.max_key - kmin;
  const int sh = max(1, 32 - __clz(range | 1u) - 10);    // CLUSTER_CELLS << sh > range
  static_assert(CLUSTER_CELLS == 1 << 10, "");
  for (int c = tid; c < CLUSTER_CELLS; c += NT) mine[c] = 0u;
  if (tid < NW * 16) wq[tid] = 0u;
  __syncthreads();
#pragma unroll 4
  for (int i = tid; i < nloc; i += NT) {
    const uint32_t key = kA[i];
    if (key != KEY_NONMEMBER) atomicAdd(&mine[(key - kmin) >> sh], 1u);
  }
  Cl<CS>::sync();
  // each CTA adds up a slice of the cells and hands it to all
  if (tid < SLICE) {
    const int c = rank * SLICE + tid;
    uint32_t t = 0u;
#pragma unroll
    for (int r = 0; r < CS; ++r) t += Cl<CS>::at(mine, r)[c];
#pragma unroll
    for (int r = 0; r < CS; ++r) Cl<CS>::at(cum, r)[c] = t;
  }
  Cl<CS>::sync();
  {
    constexpr int CPT = CLUSTER_CELLS / NT;
    uint32_t v[CPT], s = 0u;
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
      v[j] = cum[tid * CPT + j];
      s += v[j];
    }
    uint32_t run = group_excl<NT>(s, wtot, tid);
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
      cum[tid * CPT + j] = run;
      run += v[j];
    }
    if (tid == 0) cum[CLUSTER_CELLS] = (uint32_t)n_mem;
  }
  __syncthreads();
  // destinations, and the rank among the warp's members for each: a warp takes
  // consecutive candidates, so that equal radii arrive in candidate order
  const uint32_t share = (uint32_t)(n_mem + CS - 1) / CS;
  const int wchunk = ((nloc + NW * 32 - 1) / (NW * 32)) * 32;
  uint32_t* pk = ex2;                    // (the cells in it have been read)
  for (int e = warp * wchunk + lane; e - lane < min(nloc, (warp + 1) * wchunk); e += 32) {
    const uint32_t key = e < nloc ? kA[e] : KEY_NONMEMBER;
    const bool valid = key != KEY_NONMEMBER;
    uint32_t q = 0u;
    if (valid) {
      const uint32_t x = key - kmin, c = x >> sh, b = cum[c];
      q = (b + __umulhi(cum[c + 1] - b, x << (32 - sh))) / share;
    }
    unsigned peers = __ballot_sync(FULL_MASK, valid);
#pragma unroll
    for (int bit = 1; bit < CS; bit <<= 1) {
      const unsigned bb = __ballot_sync(FULL_MASK, (q & bit) != 0u);
      peers &= (q & bit) ? bb : ~bb;
    }
    const uint32_t base = wq[warp * 16 + q];
    __syncwarp();
    if (valid) {
      const unsigned below = peers & lanemask_lt();
      pk[e] = (q << 16) | (base + __popc(below));
      if (below == 0u) wq[warp * 16 + q] = base + __popc(peers);
    }
    __syncwarp();
  }
  __syncthreads();
  if (tid < CS) {
    uint32_t run = 0u;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      const uint32_t c = wq[w * 16 + tid];
      wq[w * 16 + tid] = run;
      run += c;
    }
    X.cnt[tid] = run;
  }
  Cl<CS>::sync();
  if (tid < CS) {
    uint32_t pre = 0u, tot = 0u;
#pragma unroll
    for (int r = 0; r < CS; ++r) {
      const uint32_t v = Cl<CS>::at(X.cnt, r)[tid];
      if (r < rank) pre += v;
      tot += v;
    }
    S.dpre[tid] = pre;
    S.dtot[tid] = tot;
  }
  __syncthreads();
  bool fits = true;                      // (the parts' counts take one word more than the members)
  for (int q = 0; q < CS; ++q) fits = fits && S.dtot[q] < (uint32_t)CAP;
  if (!fits) {                           // the same in every CTA
    Cl<CS>::sync();                      // every CTA has read the counts
    return -1;
  }
  for (int e = warp * wchunk + lane; e < min(nloc, (warp + 1) * wchunk); e += 32) {
    const uint32_t key = kA[e];
    if (key != KEY_NONMEMBER) {
      const uint32_t x = pk[e], q = x >> 16;
      Cl<CS>::at(reinterpret_cast<uint2*>(kB), (int)q)[S.dpre[q] + wq[warp * 16 + q] + (x & 0xffffu)] =
          make_uint2(key, vA[e]);
    }
  }
  if (tid == 0) {
    S.max_key = 0u;
    S.min_key = 0xffffffffu;
  }
  Cl<CS>::sync();
  nrec = (int)S.dtot[rank];
  uint32_t mx = 0u, mn = 0xffffffffu;
  for (int i = tid; i < nrec; i += NT) {
    const uint2 x = reinterpret_cast<const uint2*>(kB)[i];
    kA[i] = x.x;
    vA[i] = x.y;
    mx = max(mx, x.x);
    mn = min(mn, x.x);
  }
  mx = __reduce_max_sync(FULL_MASK, mx);
  mn = __reduce_min_sync(FULL_MASK, mn);
  if (lane == 0) {
    atomicMax(&S.max_key, mx);
    atomicMin(&S.min_key, mn);
  }
  __syncthreads();
  if (nrec == 0) return 0;
  if (dist_sort<NT, SORT_CELLS>(kA, vA, kB, vB, ex2, ex1, hist, wtot, vA, nrec, nrec, S.min_key, S.max_key, tid))
    return 0;
  // dozens of equal radii: the counting radix sort of this CTA's share (its
  // counters in ex1 and ex2), brought to the buffer that dist_sort leaves it in:
  // every CTA has the order in the same arrays, at whose addresses the CTAs read
  // one another's radii (Cl::at)
  static_assert(count_sort_words(NT) <= 2 * CAP, "counters fit");
  const uint32_t differ = S.max_key ^ S.min_key;
  const uint32_t diff = differ ? 0xffffffffu >> __clz(differ) : 0u;
  if (count_sort<NT, (run_length(CAP, NT) + 3) / 4 * 4>(kA, vA, kB, vB, ex1, wtot, nrec, run_length(nrec, NT), diff, 0u,
                                                        tid)) {
    for (int i = tid; i < nrec; i += NT) {
      kA[i] = kB[i];
      vA[i] = vB[i];
    }
    __syncthreads();
  }
  return 0;
}

constexpr int NT_1K = 128, NT_4K = 256, NT_8K = 512, NT_CL = 512;
template <int CAP, int CS>
constexpr int min_blocks() { return CS > 1 ? 1 : (CAP <= 1024 ? 6 : (CAP <= 4096 ? 2 : 1)); }

template <int NT, int CAP, int CT, int CS>
__global__ void __launch_bounds__(NT, (min_blocks<CAP, CS>())) unbind_kernel(OnchipLaunch L) {
  constexpr int IPT = CAP / NT;
  static_assert(IPT * NT == CAP && IPT <= 32 && (IPT & (IPT - 1)) == 0, "bad tile");
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ Smem<NT> S;
  __shared__ Xchg X;
  uint32_t* kA = (uint32_t*)dyn;
  uint32_t* vA = kA + CAP;
  uint32_t* kB = vA + CAP;
  uint32_t* vB = kB + CAP;
  float* ex1 = (float*)(vB + CAP);
  float* ex2 = ex1 + CAP;
  uint16_t* hist = (uint16_t*)(ex2 + CAP);

  const int tid = threadIdx.x, lane = tid & 31;
  const int rank = Cl<CS>::rank();
  const ParamsDev& P = L.prm;
  const bool unim = L.p.m == nullptr;                    // every particle has mass m0

  chain_open();
  for (;;) {
    if (rank == 0 && tid == 0) X.halo = atomicAdd(L.queue, 1);
    Cl<CS>::sync();
    const int hq = *Cl<CS>::at(&X.halo, 0);
    Cl<CS>::sync();
    if (hq >= L.n_halos) break;
    const HaloDev& H = L.halos[hq];
    if (tid == 0 && rank == 0) trace_mark(L.trace, H.index, 0);
    const int n_cand = (int)H.count;
    const int chunk = n_cand > 0 ? (n_cand + CS - 1) / CS : 1;
    if (chunk > CAP) {    // the scheduler never does this; report, do not overrun
      if (tid == 0 && rank == 0) atomicOr(L.out.err, ERR_CAPACITY);
      continue;
    }
    const int lo = rank * chunk;
    const int nloc = max(0, min(n_cand - lo, chunk));
    prefetch_candidates<CT>(L.p, L.out.member_idx, H.offset + lo, H.offset + lo + nloc, tid);
    if (tid == 0) {
      S.or_bits = 0u; S.and_bits = 0xffffffffu;
      S.max_m = 0u; S.max_mr = 0u; S.max_mv = 0u;
      S.max_key = 0u;
      S.min_key = 0xffffffffu;
      S.n_member = 0;
      S.acc[0] = S.acc[1] = S.acc[2] = S.acc[3] = 0;
      S.acc_n = 0; S.acc_band = 0;
    }
    __syncthreads();

    // ---- gather: key = radius bits of members, candidate position as value ----
    {
      uint32_t orb = 0u, andb = 0xffffffffu, mxm = 0u, mxr = 0u, mxv = 0u, kmx = 0u, kmn = 0xffffffffu;
      int nmem = 0;
      for (int i = tid; i < nloc; i += NT) {
        const int j = lo + i;
        const long long slot = H.offset + j;
        long long pi = slot;
        bool ok = true;
        if (L.out.member_idx) {
          pi = L.out.member_idx[slot];
          if (pi < 0 || pi >= L.p.n) { ok = false; atomicOr(L.out.err, ERR_BAD_INDEX); }
        }
        uint32_t key = KEY_NONMEMBER;
        if (ok) {
          Cand<CT> c;
          load_cand<CT>(L.p, pi, c);
          long long f[3];
          float df[3];
          cand_offset<CT>(c, H, df, f);
          if (cand_member<CT>(c, H, df, f)) {
            const float r = radius_of(df);
            key = __float_as_uint(r);
            const float m = cand_mass<CT>(L.p, c);
            float v[3];
            cand_velocity<CT>(c, v);
            if (L.rec) put_record(L.rec + 2 * (H.gbase + j), df, m, v);
            if (unim) {
              // (one mass: the maxima follow from the smallest radius and the
              // largest |v_k| below, rounding being monotone)
#pragma unroll
              for (int k = 0; k < 3; ++k) mxv = max(mxv, __float_as_uint(fabsf(v[k])));
              if (fmaxf(r, P.r_soft_f) > 0.0f) mxr = max(mxr, ~__float_as_uint(r));
            } else {
              mxm = max(mxm, __float_as_uint(fabsf(m)));
              mxr = max(mxr, __float_as_uint(fabsf(m * rinv_of(r, P.r_soft_f))));
#pragma unroll
              for (int k = 0; k < 3; ++k) mxv = max(mxv, __float_as_uint(fabsf(__fmul_rn(m, v[k]))));
            }
            ++nmem;
          }
        }
        // members start bound (removal overwrites with its iteration)
        if (L.out.removed_iter) L.out.removed_iter[slot] = key == KEY_NONMEMBER ? -1 : 0;
        kA[i] = key;
        if constexpr (CS > 1) vA[i] = (uint32_t)j;
        if (CS > 1 || key != KEY_NONMEMBER) {
          orb |= key;
          andb &= key;
        }
        if (key != KEY_NONMEMBER) {
          kmx = max(kmx, key);
          kmn = min(kmn, key);
        }
      }
      orb = __reduce_or_sync(FULL_MASK, orb);
      andb = __reduce_and_sync(FULL_MASK, andb);
      mxm = __reduce_max_sync(FULL_MASK, mxm);
      mxr = __reduce_max_sync(FULL_MASK, mxr);
      mxv = __reduce_max_sync(FULL_MASK, mxv);
      nmem = __reduce_add_sync(FULL_MASK, nmem);
      kmx = __reduce_max_sync(FULL_MASK, kmx);
      kmn = __reduce_min_sync(FULL_MASK, kmn);
      if (lane == 0) {
        atomicMax(&S.max_key, kmx);
        atomicMin(&S.min_key, kmn);
        atomicOr(&S.or_bits, orb);
        atomicAnd(&S.and_bits, andb);
        atomicMax(&S.max_m, mxm);
        atomicMax(&S.max_mr, mxr);
        atomicMax(&S.max_mv, mxv);
        atomicAdd(&S.n_member, nmem);
      }
    }
    __syncthreads();
    if constexpr (CS > 1) {
      if (tid == 0) {
        X.g_or = S.or_bits; X.g_and = S.and_bits; X.g_mxm = S.max_m; X.g_mxr = S.max_mr; X.g_mxv = S.max_mv;
        X.g_nmem = S.n_member;
        X.g_kmx = S.max_key; X.g_kmn = S.min_key;
      }
      Cl<CS>::sync();
      if (tid == 0) {
        uint32_t o = 0u, a = 0xffffffffu, m1 = 0u, m2 = 0u, m3 = 0u, kx = 0u, kn = 0xffffffffu;
        int nm = 0;
        for (int r = 0; r < CS; ++r) {
          const Xchg* Y = Cl<CS>::at(&X, r);
          o |= Y->g_or; a &= Y->g_and;
          m1 = max(m1, Y->g_mxm); m2 = max(m2, Y->g_mxr); m3 = max(m3, Y->g_mxv);
          nm += Y->g_nmem;
          kx = max(kx, Y->g_kmx); kn = min(kn, Y->g_kmn);
        }
        S.max_key = kx; S.min_key = kn;
        S.or_bits = o; S.and_bits = a; S.max_m = m1; S.max_mr = m2; S.max_mv = m3; S.n_member = nm;
      }
      __syncthreads();
    }
    const int n_mem = S.n_member;                        // members of the halo
    // the exponents of the largest m, m / r and |m v_k|
    uint32_t mxm = S.max_m, mxr = S.max_mr, mxv = S.max_mv;
    if (unim) {
      mxm = n_mem > 0 ? __float_as_uint(fabsf(L.p.m0f)) : 0u;
      mxr = mxr ? __float_as_uint(fabsf(L.p.m0f * rinv_of(__uint_as_float(~mxr), P.r_soft_f))) : 0u;
      mxv = __float_as_uint(fabsf(__fmul_rn(L.p.m0f, __uint_as_float(mxv))));
    }
    int nmem_loc = max(0, min(n_mem - lo, nloc));        // held by this CTA after the sort
    const int s_m = fix_scale(float_exponent_of_bits(mxm), n_mem);
    const int s_r = fix_scale(float_exponent_of_bits(mxr), n_mem);
    const int s_v = fix_scale(float_exponent_of_bits(mxv), n_mem);
    const long long m0fix = fix_from_float(L.p.m0f, s_m);
    // 2^-s of the mass and m/r sums as floats (0 when not normal): each
    // exact sum's float value is then one multiply, the bits of float_from_fix
    const float sc_m = pow2_neg(s_m), sc_r = pow2_neg(s_r);

    if (tid == 0 && rank == 0) trace_mark(L.trace, H.index, 1);
    // ---- radial sort (once) ----
    int which;
    if constexpr (CS == 1) {
      which = 0;
      uint32_t* aux = reinterpret_cast<uint32_t*>(ex1);    // count_sort's: ex1, ex2 and hist
      uint32_t* wtot = reinterpret_cast<uint32_t*>(&S.red[0][0]);
      // (the counts' last word, cnt[CAP], is ex2's first)
      if (n_mem > 0 && !dist_sort<NT, SORT_CELLS>(kA, vA, kB, vB, vA, reinterpret_cast<uint32_t*>(ex1),
                                                  reinterpret_cast<uint32_t*>(hist), wtot, nullptr, nloc, n_mem,
                                                  S.min_key, S.max_key, tid)) {
        for (int i = tid; i < nloc; i += NT) vA[i] = (uint32_t)i;
        uint32_t diff = S.or_bits ^ S.and_bits, sub = 0u;
        if (n_mem < n_cand) {              // non-members get a key just above the members'
          sub = S.max_key + 1u;
          diff = (S.or_bits | sub) ^ (S.and_bits & sub);
        }
        __syncthreads();
        which = count_sort<NT, (run_length(CAP, NT) + 3) / 4 * 4>(kA, vA, kB, vB, aux, wtot, nloc,
                                                                   run_length(nloc, NT), diff, sub, tid);
      }
    } else {
      which = -1;
      if (n_mem > 0)
        which = cluster_dist_sort<NT, IPT, CS>(kA, vA, kB, vB, reinterpret_cast<uint32_t*>(ex1),
                                               reinterpret_cast<uint32_t*>(ex2), reinterpret_cast<uint32_t*>(hist), S, X,
                                               nloc, n_mem, rank, nmem_loc);
      if (which < 0)
        which = cluster_radix_sort<NT, IPT, CS>(kA, vA, kB, vB, hist, S, X, nloc, chunk, S.or_bits ^ S.and_bits, rank);
    }
    if (tid == 0 && rank == 0) trace_mark(L.trace, H.index, 2);
    float* rr = (float*)(which ? kB : kA);         // radius, sorted
    uint32_t* jj = which ? vB : vA;                // candidate position
    float* mm = (float*)(which ? kA : kB);         // mass; sign bit = removed
    float* wx = (float*)(which ? vA : vB);
    float* wy = ex1;
    float* wz = ex2;

    // ---- fill: m and w = v + H d in the radial order (from the records, mostly
    // L2), each thread its own run: the exact sum m v of the members, and the
    // run's exact sums of m, m/r and its alive count
    const int ipt = run_length(nmem_loc, NT);
    const int p0 = tid * ipt;
    long long tm_own = 0, tr_own = 0, tc_own = 0;
    {
      long long smv[3] = {0, 0, 0};
      const int p1 = min(p0 + ipt, nmem_loc);
#pragma unroll 2
      for (int p = p0; p < p1; ++p) {
        const int j = (int)jj[p];
        float dfl[3], v[3], m;
        if (L.rec) {
          get_record(L.rec + 2 * (H.gbase + j), dfl, m, v);
        } else {
          const long long slot = H.offset + j;
          const long long pi = L.out.member_idx ? L.out.member_idx[slot] : slot;
          long long f[3];
          offset_of<CT>(L.p, pi, H, dfl, f);
          load_velocity<CT>(L.p, pi, v);
          m = load_mass<CT>(L.p, pi);
        }
        // with a uniform mass the slot holds 1 / max(r, r_soft) instead (the
        // mass is m0): the reciprocal is formed once, not every iteration
        const float ri = rinv_of(rr[p], P.r_soft_f);
        mm[p] = unim ? ri : m;
        wx[p] = fmaf(P.Hf, dfl[0], v[0]);
        wy[p] = fmaf(P.Hf, dfl[1], v[1]);
        wz[p] = fmaf(P.Hf, dfl[2], v[2]);
        tm_own += unim ? m0fix : fix_from_float(m, s_m);
        tr_own += fix_from_float(m * ri, s_r);
#pragma unroll
        for (int k = 0; k < 3; ++k) smv[k] += fix_from_float(__fmul_rn(m, v[k]), s_v);
      }
      tc_own = max(0, p1 - p0);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const long long t = warp_sum(smv[k]);
        if (lane == 0 && t != 0) atomicAdd((unsigned long long*)&S.acc[k], (unsigned long long)t);
      }
    }
    __syncthreads();
    if constexpr (CS > 1) {
      if (tid == 0) { X.mv[0] = S.acc[0]; X.mv[1] = S.acc[1]; X.mv[2] = S.acc[2]; }
      Cl<CS>::sync();
      if (tid < 3) {
        long long t = 0;
        for (int r = 0; r < CS; ++r) t += Cl<CS>::at(&X.mv[0], r)[tid];
        S.mv[tid] = t;
      }
    } else {
      if (tid < 3) S.mv[tid] = S.acc[tid];
    }
    __syncthreads();

    if (tid == 0 && rank == 0) trace_mark(L.trace, H.index, 3);
    // ---- iterate (Appendix A) ----
    int n_iter = 0, status = 0;
    long long part_iter = 0, n_band = 0;
    int n_alive = n_mem;
    bool converged = false;
    // one CTA: every thread keeps the exact sum m v and forms v_bulk itself
    // (the same bits in every thread), and the removal sums alternate
    // between two buffers, so an iteration takes three barriers
    long long mvl[3] = {S.mv[0], S.mv[1], S.mv[2]};
    float vbl[3] = {0.0f, 0.0f, 0.0f};
    if constexpr (CS == 1) {
      if (tid == 0)
        for (int bsel = 0; bsel < 2; ++bsel) {
          S.racc[bsel][0] = S.racc[bsel][1] = S.racc[bsel][2] = S.racc[bsel][3] = 0;
          S.racc_n[bsel] = 0;
          S.racc_band[bsel] = 0;
        }
    }
    // a cluster: one exchange per iteration (cluster_exchange) carries the
    // scan totals of the current set and the previous iteration's removals;
    // the last one, of the final set, also serves the emit
    long long e_tm = 0, e_tr = 0, e_tc = 0;   // the emit's prefixes
    int xs = 0;
    for (;;) {
      long long tm = tm_own, tr = tr_own;
      long long T_tot;
      int bsel = 0;
      if constexpr (CS == 1) {
        if (!(n_alive > 0 && n_iter < P.max_iter)) break;
        ++n_iter;
        part_iter += n_alive;
        bsel = n_iter & 1;
        block_exclusive_scan2<NT>(tm, tr, S);
        T_tot = S.tot[1];
        // v_bulk = sum m v / sum m of the current set, from the exact sums
        // (with AHF_VAR_VBULK_INITIAL the first iteration's value is kept)
        if (n_iter == 1 || !P.vbulk_initial) {
          const float mt = float_from_fix(S.tot[0], s_m);
          vbl[0] = float_from_fix(mvl[0], s_v) / mt;
          vbl[1] = float_from_fix(mvl[1], s_v) / mt;
          vbl[2] = float_from_fix(mvl[2], s_v) / mt;
        }
        if (tid == 0) {                  // the next iteration's buffer: its readers are past the scan
          S.racc[bsel ^ 1][0] = S.racc[bsel ^ 1][1] = S.racc[bsel ^ 1][2] = S.racc[bsel ^ 1][3] = 0;
          S.racc_n[bsel ^ 1] = 0;
          S.racc_band[bsel ^ 1] = 0;
        }
      } else {
        long long tc = tc_own;
        block_exclusive_scan3<NT>(tm, tr, tc, S);
        cluster_exchange<NT, CS>(S, X, rank, xs, n_iter == 0);
        xs ^= 1;
        bool stop = false;
        if (n_iter > 0) {                // the previous iteration's removals
          const int removed = S.c_removed;
          n_band += S.c_band;
          n_alive -= removed;
          if (removed == 0) {
            converged = true;
            stop = true;
          }
        }
        if (stop || !(n_alive > 0 && n_iter < P.max_iter)) {
          e_tm = tm;
          e_tr = tr;
          e_tc = tc;
          break;
        }
        ++n_iter;
        part_iter += n_alive;
        if (tid == 0) {
          if (n_iter == 1 || !P.vbulk_initial) {
            const float mt = float_from_fix(S.c_tot[0], s_m);
            S.vb[0] = float_from_fix(S.mv[0], s_v) / mt;
            S.vb[1] = float_from_fix(S.mv[1], s_v) / mt;
            S.vb[2] = float_from_fix(S.mv[2], s_v) / mt;
          }
          S.acc[0] = S.acc[1] = S.acc[2] = S.acc[3] = 0;
          S.acc_n = 0;
          S.acc_band = 0;
        }
        __syncthreads();
        tm += S.c_pre[0];
        tr += S.c_pre[1];
        T_tot = S.c_tot[1];
        vbl[0] = S.vb[0];
        vbl[1] = S.vb[1];
        vbl[2] = S.vb[2];
      }
      const float vb0 = vbl[0], vb1 = vbl[1], vb2 = vbl[2];
      long long rm = 0, rq = 0, rv0 = 0, rv1 = 0, rv2 = 0;
      int nrem = 0, nband = 0;
      uint32_t rmask = 0;                 // this thread's removals (bit k: position p0 + k)
      const int run = min(ipt, nmem_loc - p0);            // members of this thread's run
      if (sc_m != 0.0f && sc_r != 0.0f) {
        if (unim)
          member_pass<0>(rr, mm, wx, wy, wz, p0, run, P, true, L.p.m0f, m0fix, s_m, s_r, sc_m, sc_r, vb0, vb1, vb2, tm,
                         T_tot - tr, rmask, nband);
        else
          member_pass<1>(rr, mm, wx, wy, wz, p0, run, P, false, 0.0f, 0ll, s_m, s_r, sc_m, sc_r, vb0, vb1, vb2, tm,
                         T_tot - tr, rmask, nband);
      } else {
        member_pass<2>(rr, mm, wx, wy, wz, p0, run, P, unim, L.p.m0f, m0fix, s_m, s_r, 0.0f, 0.0f, vb0, vb1, vb2, tm,
                       T_tot - tr, rmask, nband);
      }
      // the removed: their mark, their exact terms, m v from the stored velocity,
      // and their record
      for (uint32_t b = rmask; b; b &= b - 1) {
        const int q = p0 + __ffs(b) - 1;
        const float mq = mm[q];
        mm[q] = -mq;
        const float m = unim ? L.p.m0f : mq;
        const float ri = unim ? mq : rinv_of(rr[q], P.r_soft_f);
        rm += unim ? m0fix : fix_from_float(m, s_m);
        rq += fix_from_float(m * ri, s_r);
        const int j = (int)jj[q];
        const long long slot = H.offset + j;
        float v[3];
        if (L.rec) get_velocity_record(L.rec + 2 * (H.gbase + j), v);
        else load_velocity<CT>(L.p, L.out.member_idx ? L.out.member_idx[slot] : slot, v);
        rv0 += fix_from_float(__fmul_rn(m, v[0]), s_v);
        rv1 += fix_from_float(__fmul_rn(m, v[1]), s_v);
        rv2 += fix_from_float(__fmul_rn(m, v[2]), s_v);
        if (L.out.removed_iter) L.out.removed_iter[slot] = n_iter;
        ++nrem;
      }
      tm_own -= rm;
      tr_own -= rq;
      tc_own -= nrem;
      nrem = __reduce_add_sync(FULL_MASK, nrem);
      nband = __reduce_add_sync(FULL_MASK, nband);
      long long* acc = CS == 1 ? S.racc[bsel] : S.acc;
      int* acc_n = CS == 1 ? &S.racc_n[bsel] : &S.acc_n;
      int* acc_band = CS == 1 ? &S.racc_band[bsel] : &S.acc_band;
      if (nrem) {
        rm = warp_sum(rm); rv0 = warp_sum(rv0); rv1 = warp_sum(rv1); rv2 = warp_sum(rv2);
        if (lane == 0) {
          atomicAdd((unsigned long long*)&acc[0], (unsigned long long)rm);
          atomicAdd((unsigned long long*)&acc[1], (unsigned long long)rv0);
          atomicAdd((unsigned long long*)&acc[2], (unsigned long long)rv1);
          atomicAdd((unsigned long long*)&acc[3], (unsigned long long)rv2);
        }
      }
      if (lane == 0 && (nrem | nband)) {
        atomicAdd(acc_n, nrem);
        atomicAdd(acc_band, nband);
      }
      __syncthreads();
      if constexpr (CS == 1) {
        const int removed = *acc_n;
        n_band += *acc_band;
        mvl[0] -= acc[1];
        mvl[1] -= acc[2];
        mvl[2] -= acc[3];
        n_alive -= removed;
        if (removed == 0) {              // the scan was of the final set
          converged = true;
          e_tm = tm;
          e_tr = tr;
          break;
        }
      }
      // a cluster: this iteration's removal sums go out with the next exchange
    }
    if (n_alive == 0) status |= AHF_HALO_EMPTY;
    else if (!converged) status |= AHF_HALO_NOT_CONVERGED;
    if constexpr (CS == 1) {
      if (tid == 0) {                    // for the record (the emit's scan barriers order it)
        S.mv[0] = mvl[0];
        S.mv[1] = mvl[1];
        S.mv[2] = mvl[2];
      }
    }

    if (tid == 0 && rank == 0) trace_mark(L.trace, H.index, 4);
    // ---- emit: bound list, phi, compacted (r, inclusive M) for the virial search ----
    // (a uniform mass needs no masses: the bound list and phi are compacted
    // there and go out coalesced, instead of 32 sectors per warp and store)
    float* rc = wx;                       // reuse: w is no longer needed
    long long* mc = (long long*)ex1;      // ex1 and ex2 are contiguous
    float* pc = ex1;                      // uniform mass: phi, candidate position
    uint32_t* jc = (uint32_t*)ex2;
    {
      long long tm = tm_own, tr = tr_own, tc = tc_own;
      if constexpr (CS == 1) {
        if (converged) {
          tm = e_tm;
          tr = e_tr;
          tc = group_excl<NT>((uint32_t)tc_own, reinterpret_cast<uint32_t*>(&S.red[0][0]), tid);
          if (tid < 3) S.c_tot[tid] = tid < 2 ? S.tot[tid] : n_alive;
        } else {
          block_exclusive_scan3<NT>(tm, tr, tc, S);
          if (tid < 3) S.c_tot[tid] = S.tot[tid];
        }
        if (tid < 3) S.c_pre[tid] = 0;
        __syncthreads();
      } else {                            // the last exchange was of the final set
        tm = e_tm;
        tr = e_tr;
        tc = e_tc;
      }
      const long long C_pre = S.c_pre[2];
      const long long C_loc = CS == 1 ? S.c_tot[2] : S.tot[2];
      const long long T_tot = S.c_tot[1];
      const long long nb = S.c_tot[2];
      tm += S.c_pre[0];
      tr += S.c_pre[1];
      long long tl = tc;                  // local rank of the thread's first bound particle
      long long out = T_tot - tr;
      const int p1 = min(p0 + ipt, nmem_loc);
      for (int q = p0; q < p1; ++q) {
        const float mq = mm[q];
        if (!signbit(mq)) {
          const float r = rr[q];
          const float m = unim ? L.p.m0f : mq;
          const float ri = unim ? mq : rinv_of(r, P.r_soft_f);
          const long long mfix = (unim ? m0fix : fix_from_float(m, s_m));
          const float phi = phi_of(fix_to_float_fast(tm, s_m, sc_m), ri, fix_to_float_fast(out, s_r, sc_r), P.Gf);
          const int j = (int)jj[q];
          rc[tl] = r;
          if (unim) {
            pc[tl] = phi;
            jc[tl] = (uint32_t)j;
          } else {
            const long long slot = H.offset + j;
            const long long dst = H.offset + C_pre + tl;
            L.out.bound_idx[dst] = L.out.member_idx ? L.out.member_idx[slot] : slot;
            if (L.out.phi) ((float*)L.out.phi)[dst] = phi;
            mc[tl] = tm + mfix;
          }
          tm += mfix;
          out -= fix_from_float(m * ri, s_r);
          tl += 1;
        }
      }
      if (tid == 0) S.k_first = 0x7fffffff;
      __syncthreads();
      if (unim) {
        const long long d0 = H.offset + C_pre;
        for (int i = tid; i < (int)C_loc; i += NT) {
          const long long slot = H.offset + (long long)jc[i];
          L.out.bound_idx[d0 + i] = L.out.member_idx ? L.out.member_idx[slot] : slot;
          if (L.out.phi) ((float*)L.out.phi)[d0 + i] = pc[i];
        }
      }
      float r_after = __int_as_float(0x7f800000);   // +inf: radius of the next bound particle
      if constexpr (CS > 1) {
        if (tid == 0) {
          X.nb_loc = (int)C_loc;
          X.first_r = C_loc > 0 ? rc[0] : 0.0f;
        }
        Cl<CS>::sync();
        for (int r2 = rank + 1; r2 < CS; ++r2) {
          const Xchg* Y = Cl<CS>::at(&X, r2);
          if (Y->nb_loc > 0) { r_after = Y->first_r; break; }
        }
      }
      // virial: first k with M_k < delta_rho 4pi/3 r_{k+1}^3 (r_{N+1} = inf)
      int kf = 0x7fffffff;
      for (int k = 0; k < ipt; ++k) {
        const int kk = p0 + k;
        if (kk < C_loc) {
          const float rn = kk + 1 < C_loc ? rc[kk + 1] : r_after;
          bool cross = true;
          if (!isinf(rn)) {
            const long long mk = unim ? (C_pre + kk + 1) * m0fix : mc[kk];
            const float lhs = fix_to_float_fast(mk, s_m, sc_m);
            const float rhs = P.crit_f * rn * rn * rn;
            if (lhs < rhs * (1.0f - 1e-5f)) cross = true;
            else if (lhs > rhs * (1.0f + 1e-5f)) cross = false;
            else {
              const double rd = (double)rn;
              cross = double_from_fix(mk, s_m) < P.crit * rd * rd * rd;
            }
          }
          if (cross) { kf = (int)(C_pre + kk); break; }
        }
      }
      kf = (int)__reduce_min_sync(FULL_MASK, (unsigned)kf);
      if (lane == 0 && kf != 0x7fffffff) atomicMin(&S.k_first, kf);
      __syncthreads();
      if constexpr (CS > 1) {
        if (tid == 0) X.kf = S.k_first;
        Cl<CS>::sync();
        if (tid == 0) {
          int k = 0x7fffffff;
          for (int r2 = 0; r2 < CS; ++r2) k = min(k, Cl<CS>::at(&X, r2)->kf);
          S.k_first = k;
        }
        __syncthreads();
      }
      // the CTA holding the crossing particle writes the record
      const int k = S.k_first;
      const bool owner = nb > 0 ? (k >= C_pre && k < C_pre + C_loc) : rank == 0;
      if (owner) {
        // the record, its FP64 parts spread over the first thread of four
        // warps (one per SM sub-partition): the virial pair, and one bulk
        // velocity component each
        ahf_result* R = L.out.res + H.index;
        if (tid == 0) {
          long long kv = -1;
          double mv = 0.0, rv = 0.0;
          if (nb > 0) {
            const int kl = (int)(k - C_pre);
            // M_vir: (k+1) m0 in FP64 for a uniform mass, else the exact sum
            const long long mkx = unim ? 0 : mc[kl];
            const double mk = unim ? (double)(k + 1) * L.p.m0 : double_from_fix(mkx, s_m);
            const float mkf = unim ? (float)(k + 1) * L.p.m0f : float_from_fix(mkx, s_m);
            if (k == nb - 1) status |= AHF_HALO_RVIR_BEYOND_EDGE;
            if (below_threshold(mk, mkf, rc[kl], P.crit_f, P.crit)) {
              status |= AHF_HALO_RVIR_NONE;
            } else {
              kv = k;
              mv = mk;
              rv = virial_radius(mk, P.inv_crit);
              if (P.rise_edge && k == nb - 1) {
                // bound position p of the cluster: rank q holds [pre_q, pre_q + nb_loc_q)
                auto at = [&](long long p, double& r, double& m) {
                  int q = 0;
                  long long pre = 0;
                  if constexpr (CS > 1) {
                    for (; q < CS - 1; ++q) {
                      const long long nl = Cl<CS>::at(&X, q)->nb_loc;
                      if (p < pre + nl) break;
                      pre += nl;
                    }
                  }
                  const int l = (int)(p - pre);
                  r = float_to_double(Cl<CS>::at(rc, q)[l]);
                  m = unim ? (double)(p + 1) * L.p.m0 : double_from_fix(Cl<CS>::at(mc, q)[l], s_m);
                };
                const long long ke = rise_edge_index(nb, at);
                if (ke >= 0) {
                  at(ke, rv, mv);
                  kv = ke;
                  status |= AHF_HALO_RISE_EDGE;
                }
              }
            }
          }
          R->n_bound = nb;
          R->n_member = n_mem;
          R->part_iter = part_iter;
          R->n_band = n_band;
          R->k_vir = kv;
          R->n_iter = n_iter;
          R->status = status;
          R->m_vir = mv;
          R->r_vir = rv;
          S.rvir = rv;
          S.kvir = kv;
          if constexpr (CS > 1) {
#pragma unroll
            for (int r2 = 0; r2 < CS; ++r2) Cl<CS>::at(&X, r2)->rvir = rv;
          }
        } else if (tid == 32 || tid == 64 || tid == 96) {
          const int c = tid / 32 - 1;
          R->vbulk[c] = nb > 0 ? quotient(double_from_fix(S.mv[c], s_v), double_from_fix(S.c_tot[0], s_m)) : 0.0;
        }
      }
      if constexpr (CS > 1) {
        if (L.rows.prof && L.rows.n_bins <= FUSE_BINS) {
          // rows of a halo spread over the cluster: each CTA counts its share of
          // the radial order at every edge and adds that to rank 0's counts; the
          // inclusive mass is the largest CTA's (the last particle's inside)
          if (rank == 0)
            for (int b = tid; b <= L.rows.n_bins; b += NT) X.pc[b] = 0;
          if (tid < CS && C_loc > 0 && C_pre + C_loc == nb) Cl<CS>::at(&X, tid)->last_r = rc[(int)C_loc - 1];
          Cl<CS>::sync();
          const double r_vir = X.rvir;
          const double r_out = r_vir > 0.0 ? r_vir : (nb > 0 ? (double)X.last_r : 0.0);
          const float r_out_f = (float)r_out;
          const int n = L.rows.n_bins;
          for (int b = tid; b <= n; b += NT) {
            const int lo = count_inside(rc, [](int k) { return k; }, (int)C_loc,
                                        b == n ? r_out_f : r_out_f * L.rows.factor_f[b], r_out,
                                        b == n ? 1.0 : L.rows.factor[b]);
            if (lo > 0) atomicAdd(&Cl<CS>::at(&X, 0)->pc[b], lo);
            if (!unim) X.pm[b] = lo > 0 ? mc[lo - 1] : 0;
          }
          Cl<CS>::sync();
          if (rank == 0) {
            double* out = L.rows.prof + (size_t)H.index * n * 4;
            const float inv_r = 1.0f / r_out_f;
            for (int b = tid; b < n; b += NT) {
              const long long c0 = X.pc[b], c1 = X.pc[b + 1];
              long long f0 = 0, f1 = 0;
              if (!unim) {
#pragma unroll
                for (int r2 = 0; r2 < CS; ++r2) {
                  const Xchg* Y = Cl<CS>::at(&X, r2);
                  f0 = max(f0, Y->pm[b]);
                  f1 = max(f1, Y->pm[b + 1]);
                }
              }
              if (nb == 0) {
                out[4 * b + 0] = out[4 * b + 1] = out[4 * b + 2] = out[4 * b + 3] = 0.0;
                continue;
              }
              double M1, Ms;
              if (unim) {
                M1 = (double)c1 * L.p.m0;
                Ms = (double)(c1 - c0) * L.p.m0;
              } else {
                M1 = double_from_fix(f1, s_m);
                Ms = double_from_fix(f1 - f0, s_m);
              }
              out[4 * b + 0] = (double)(c1 - c0);
              out[4 * b + 1] = M1;
              out[4 * b + 2] = shell_density(Ms, r_out, inv_r, L.rows.factor, L.rows.factor_f, n, b);
              out[4 * b + 3] = circular_velocity(P.G, P.Gf, M1, r_out, inv_r, L.rows.factor, L.rows.factor_f, n, b);
            }
          }
        }
      }
      if constexpr (CS == 1) {
        if (L.rows.prof) {
          __syncthreads();                        // S.rvir
          profile_rows(L.rows, H.index, rc, mc, [](long long kk) { return (int)kk; }, nb, S.rvir, S.kvir, s_m,
                       P.G, P.Gf, unim ? &L.p.m0 : nullptr, tid, NT);
        }
      }
    }
    if (tid == 0 && rank == 0 && L.trace) {
      long long* t = L.trace + (size_t)H.index * AHF_TRACE_FIELDS;
      t[5] = global_ns();
      t[6] = sm_id();
      t[7] = L.variant + 256ll * n_iter;
    }
    Cl<CS>::sync();
  }
  if (tid == 0 && rank == 0) chain_close(L.done, (int)gridDim.x / CS);
}

// Dynamic shared memory: six 4-byte arrays of CAP slots, then the sort's
// counters (per-warp digit counts in a cluster, dist_sort's cells in one CTA).
template <int NT, int CAP, int CS>
constexpr size_t dyn_bytes() {
  constexpr int words = SORT_CELLS + 8;
  static_assert(CS > 1 || count_sort_words(NT) <= 2 * CAP + words, "count_sort's counters lie in ex1, ex2 and hist");
  return (size_t)CAP * 24 + (CS == 1 ? (size_t)words * 4 : (size_t)(NT / 32) * 256 * 2);
}

template <int CS>
void cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr) {
  cfg.attrs = attr;
  cfg.numAttrs = 0;
  if (CS == 1) return;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CS;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.numAttrs = 1;
}

template <int NT, int CAP, int CT, int CS>
cudaError_t launch_variant(const OnchipLaunch& L, int grid, cudaStream_t s) {
  auto k = unbind_kernel<NT, CAP, CT, CS>;
  constexpr size_t smem = dyn_bytes<NT, CAP, CS>();
  static std::atomic<unsigned long long> attrs_set{0};
  if (first_use_on_device(attrs_set)) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (CS > 8) {
      e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e != cudaSuccess) return e;
    }
    mark_used_on_device(attrs_set);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3(NT, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  cluster_config<CS>(cfg, attr);
  if (L.follow) follow_config(cfg, attr);
  return cudaLaunchKernelEx(&cfg, k, L);
}

// CTAs of the variant that can be resident at once (whole clusters only).
template <int NT, int CAP, int CS>
int max_grid_variant(int device) {
  auto k = unbind_kernel<NT, CAP, AHF_COORD_F32_REL, CS>;
  constexpr size_t smem = dyn_bytes<NT, CAP, CS>();
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  if constexpr (CS == 1) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, NT, smem) != cudaSuccess || per_sm < 1) {
      cudaGetLastError();
      per_sm = 1;
    }
    return per_sm * sms;
  } else {
    if (CS > 8) cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(CS * (sms / CS)), 1, 1);
    cfg.blockDim = dim3(NT, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    cluster_config<CS>(cfg, attr);
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, k, &cfg) != cudaSuccess) {
      cudaGetLastError();
      clusters = 0;
    }
    return clusters * CS;
  }
}

}  // namespace

// Variants: 0 = 1 CTA x 128 threads / 1024 slots, 1 = 1 x 256 / 4096,
// 2 = 1 x 512 / 8192, 3/4/5/6 = clusters of 2/4/8/16 CTAs x 512 / 8192 slots.
int onchip_cluster_size(int variant) {
  switch (variant) {
    case 3: return 2;
    case 4: return 4;
    case 5: return 8;
    case 6: return 16;
    default: return 1;
  }
}

int onchip_capacity(int variant) {
  switch (variant) {
    case 0: return 1024;
    case 1: return 4096;
    case 2: return 8192;
    case 3: return 2 * 8192;
    case 4: return 4 * 8192;
    case 5: return 8 * 8192;
    case 6: return 16 * 8192;
    default: return 0;
  }
}

int onchip_max_grid(int variant, int device) {
  switch (variant) {
    case 0: return max_grid_variant<NT_1K, 1024, 1>(device);
    case 1: return max_grid_variant<NT_4K, 4096, 1>(device);
    case 2: return max_grid_variant<NT_8K, 8192, 1>(device);
    case 3: return max_grid_variant<NT_CL, 8192, 2>(device);
    case 4: return max_grid_variant<NT_CL, 8192, 4>(device);
    case 5: return max_grid_variant<NT_CL, 8192, 8>(device);
    case 6: return max_grid_variant<NT_CL, 8192, 16>(device);
    default: return 0;
  }
}

cudaError_t launch_onchip(const OnchipLaunch& L, int variant, int grid, cudaStream_t s) {
  const bool f64 = L.p.coord_type == AHF_COORD_F64;
  switch (variant) {
    case 0: return f64 ? launch_variant<NT_1K, 1024, AHF_COORD_F64, 1>(L, grid, s)
                       : launch_variant<NT_1K, 1024, AHF_COORD_F32_REL, 1>(L, grid, s);
    case 1: return f64 ? launch_variant<NT_4K, 4096, AHF_COORD_F64, 1>(L, grid, s)
                       : launch_variant<NT_4K, 4096, AHF_COORD_F32_REL, 1>(L, grid, s);
    case 2: return f64 ? launch_variant<NT_8K, 8192, AHF_COORD_F64, 1>(L, grid, s)
                       : launch_variant<NT_8K, 8192, AHF_COORD_F32_REL, 1>(L, grid, s);
    case 3: return f64 ? launch_variant<NT_CL, 8192, AHF_COORD_F64, 2>(L, grid, s)
                       : launch_variant<NT_CL, 8192, AHF_COORD_F32_REL, 2>(L, grid, s);
    case 4: return f64 ? launch_variant<NT_CL, 8192, AHF_COORD_F64, 4>(L, grid, s)
                       : launch_variant<NT_CL, 8192, AHF_COORD_F32_REL, 4>(L, grid, s);
    case 5: return f64 ? launch_variant<NT_CL, 8192, AHF_COORD_F64, 8>(L, grid, s)
                       : launch_variant<NT_CL, 8192, AHF_COORD_F32_REL, 8>(L, grid, s);
    case 6: return f64 ? launch_variant<NT_CL, 8192, AHF_COORD_F64, 16>(L, grid, s)
                       : launch_variant<NT_CL, 8192, AHF_COORD_F32_REL, 16>(L, grid, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace ahf
