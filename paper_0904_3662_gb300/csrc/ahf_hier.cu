// Hosts and subhaloes in dependency order (Sect. 2.1): the kernels around
// each level's unbinding.
//
// A level is unbound with member lists that leave out the candidates a
// descendant already bound: `owner` holds, per particle, the last halo that
// bound it (level rank in the high 32 bits, halo index in the low 32, so an
// atomic maximum keeps the latest level and, within a level, the highest
// index); `anc` maps every deeper halo to its ancestor on the current level.
// The level's results land in scratch (records by level position, removal
// iterations by compacted slot) and are scattered to the caller's arrays.
//
// A level's haloes are cut into chunks of HIER_CHUNK candidates, one CTA each: a
// host has 1e5 to 1e7 candidates and its level few haloes, and one CTA per halo
// left the chip idle (9 hosts of 5e5 candidates in all and 180 subhaloes:
// 404 us a level to compact and 304 us to scatter, 25 and 14 us in chunks).  A
// chunk's first compacted position is the sum of the counts of its halo's
// earlier chunks, which the counting kernel left.
#include <cstdint>

#include "ahf_device.cuh"

namespace ahf {
namespace {

constexpr int PT = 256;

// Particle of candidate slot `slot` of halo h, and whether the halo keeps it.
__device__ __forceinline__ bool kept_candidate(const HierLaunch& L, int h, long long slot, long long& q) {
  q = L.member_idx ? L.member_idx[slot] : slot;
  if (q < 0 || q >= L.n_particles) return true;   // left to the unbinding, which reports the bad index
  const long long own = L.owner[q];
  const int t = own >= 0 ? (int)(own & 0xffffffffll) : -1;
  return !(t >= 0 && L.anc[t] == h);
}

// Kept candidates of each chunk.
__global__ void __launch_bounds__(PT) hier_count(HierLaunch L) {
  __shared__ int red[PT / 32];
  const int c = blockIdx.x;
  const int h = L.level[L.chunk_level[c]];
  const long long off = L.halos[h].offset, cnt = L.halos[h].count;
  const long long s0 = (long long)L.chunk_ord[c] * HIER_CHUNK, s1 = min(s0 + HIER_CHUNK, cnt);
  int n = 0;
  for (long long j = s0 + threadIdx.x; j < s1; j += PT) {
    long long q;
    n += kept_candidate(L, h, off + j, q) ? 1 : 0;
  }
  n = __reduce_add_sync(FULL_MASK, n);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = n;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int w = 0; w < PT / 32; ++w) t += red[w];
    L.chunk_kept[c] = t;
  }
}

// The kept candidates, compacted in slot order; cand_map: each candidate's
// compacted position, -1 when dropped.
__global__ void __launch_bounds__(PT) hier_compact(HierLaunch L) {
  __shared__ int wsum[2][PT / 32];
  __shared__ long long red[PT / 32];
  const int c = blockIdx.x, ord = L.chunk_ord[c];
  const int i = L.chunk_level[c];
  const int h = L.level[i];
  const long long off = L.halos[h].offset, cnt = L.halos[h].count;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  long long base = 0;
  for (int k = c - ord + (int)threadIdx.x; k < c; k += PT) base += L.chunk_kept[k];
  base = warp_sum(base);
  if (lane == 0) red[warp] = base;
  __syncthreads();
  base = 0;
  for (int w = 0; w < PT / 32; ++w) base += red[w];
  const long long s0 = (long long)ord * HIER_CHUNK, s1 = min(s0 + HIER_CHUNK, cnt);
  if (threadIdx.x == 0 && s1 == cnt) L.kept[i] = base + L.chunk_kept[c];
  int turn = 0;
  for (long long r = s0; r < s1; r += PT, turn ^= 1) {
    const long long j = r + threadIdx.x;
    long long q = -1;
    const bool keep = j < s1 && kept_candidate(L, h, off + j, q);
    const unsigned b = __ballot_sync(FULL_MASK, keep);
    if (lane == 0) wsum[turn][warp] = __popc(b);
    __syncthreads();                     // (the other half is free again after the next round's)
    int before = 0, total = 0;
    for (int w = 0; w < PT / 32; ++w) {
      if (w < warp) before += wsum[turn][w];
      total += wsum[turn][w];
    }
    const long long pos = base + before + __popc(b & lanemask_lt());
    if (keep) L.members[off + pos] = q;
    if (j < s1) L.cand_map[off + j] = keep ? pos : -1;
    base += total;
  }
}

// The level's records, removal iterations by candidate slot, and the owner
// marks of its bound particles, one CTA per chunk of slots.
__global__ void __launch_bounds__(PT) hier_scatter(HierLaunch L) {
  const int c = blockIdx.x, ord = L.chunk_ord[c];
  const int i = L.chunk_level[c];
  const int h = L.level[i];
  const long long off = L.halos[h].offset, cnt = L.halos[h].count;
  const long long s0 = (long long)ord * HIER_CHUNK, s1 = min(s0 + HIER_CHUNK, cnt);
  if (threadIdx.x == 0 && ord == 0) L.res[h] = L.res_level[i];
  const long long n_bound = L.res_level[i].n_bound;
  const long long tag = ((long long)L.rank << 32) | (long long)h;
  for (long long j = s0 + threadIdx.x; j < s1; j += PT) {
    if (L.removed_iter) {
      const long long m = L.cand_map[off + j];
      L.removed_iter[off + j] = m >= 0 ? L.rem_level[off + m] : -1;
    }
    if (j < n_bound) {
      const long long q = L.bound_idx[off + j];
      if (q >= 0 && q < L.n_particles) atomicMax((long long*)&L.owner[q], tag);
    }
  }
}

}  // namespace

cudaError_t launch_hier_compact(const HierLaunch& L, int n_chunks, cudaStream_t s) {
  if (n_chunks > 0) {
    hier_count<<<n_chunks, PT, 0, s>>>(L);
    hier_compact<<<n_chunks, PT, 0, s>>>(L);
  }
  return cudaGetLastError();
}

cudaError_t launch_hier_scatter(const HierLaunch& L, int n_chunks, cudaStream_t s) {
  if (n_chunks > 0) hier_scatter<<<n_chunks, PT, 0, s>>>(L);
  return cudaGetLastError();
}

}  // namespace ahf
