// The few largest entries of a row that is streamed once by one CTA or a cluster: a list in shared memory of the
// entries above a running threshold, cut back to its best by counting ranks.  Used by the draft sampler
// (entries: Gumbel keys) and the dynamic-tree expansion (entries: pre-softmax values).
#pragma once

#include "verify_stream.cuh"

namespace lantern {
namespace stream {

constexpr int kIterElems = 4096;                 // row elements one CTA handles between two barriers
constexpr int kListCap = kIterElems + 256;       // candidate entries
constexpr int kExtra = 4;                        // the list is cut back to s + kExtra entries
constexpr int kMaxR = LANTERN_MAX_CHILDREN + kExtra;
constexpr int kFinal = kMaxCluster * kMaxR;      // candidates of all CTAs of a row

__device__ __forceinline__ bool key_before(float ka, int ia, float kb, int ib) {   // a ranks before b
  return ka > kb || (ka == kb && ia < ib);
}
__device__ __forceinline__ void warp_key_first(float& k, int& i) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float ok = __shfl_xor_sync(0xffffffffu, k, o);
    const int oi = __shfl_xor_sync(0xffffffffu, i, o);
    if (key_before(ok, oi, k, i)) { k = ok; i = oi; }
  }
}

struct TopList {
  uint2* list;      // [kListCap] (key bits, token); entries that only passed the test of the pass hold z bits instead
  int* cnt;         // entries in the list
  uint2* fin;       // [kFinal] candidates of all CTAs of the row (key bits, token), in CTA 0
  double* fkey;     // [kFinal] their exact keys
  uint2* pk;        // [2][SW] warps' best entries of a selection round
  uint2* top;       // [16] winners of the rounds of a cut
  uint2* rinfo;     // [kMaxCluster] per CTA of the row: number of candidates, T (in CTA 0)
};

// Cut the list back to its R best entries (key descending, token ascending).  Returns the new
// threshold: the key of the R-th entry, or `T` unchanged when the list has fewer than R entries.
__device__ __forceinline__ float cut_list(const TopList& s, int R, float T) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = min(*s.cnt, kListCap);
  float pk = INFINITY;
  int pt = -1;
  int got = 0;
  for (int round = 0; round < R; ++round) {
    float bk = -INFINITY;
    int bt = 0x7fffffff;
    for (int i = tid; i < n; i += ST) {
      const uint2 en = s.list[i];
      const float k = __uint_as_float(en.x);
      const int t = static_cast<int>(en.y);
      if (key_before(pk, pt, k, t) && key_before(k, t, bk, bt)) { bk = k; bt = t; }
    }
    warp_key_first(bk, bt);
    uint2* buf = s.pk + (round & 1) * SW;
    if (lane == 0) buf[warp] = make_uint2(__float_as_uint(bk), static_cast<uint32_t>(bt));
    __syncthreads();
    float ck = -INFINITY;
    int ct = 0x7fffffff;
    if (lane < SW) { ck = __uint_as_float(buf[lane].x); ct = static_cast<int>(buf[lane].y); }
    warp_key_first(ck, ct);
    if (ct == 0x7fffffff) break;                 // fewer than R entries (the same in every thread)
    if (tid == 0) s.top[round] = make_uint2(__float_as_uint(ck), static_cast<uint32_t>(ct));
    pk = ck;
    pt = ct;
    ++got;
  }
  __syncthreads();                               // every scan of the list is over
  if (tid < got) s.list[tid] = s.top[tid];
  if (tid == 0) *s.cnt = got;
  __syncthreads();
  return got == R ? pk : T;
}

// The same cut for a list of at most ST entries: every thread counts how many entries rank before its
// own, so there is no chain of selection rounds.
__device__ __forceinline__ float cut_ranked(const TopList& s, int R, float T) {
  const int tid = threadIdx.x, n = *s.cnt;
  float k = -INFINITY;
  int t = 0x7fffffff, rank = 0;
  if (tid < n) {
    const uint2 en = s.list[tid];
    k = __uint_as_float(en.x);
    t = static_cast<int>(en.y);
#pragma unroll 8
    for (int i = 0; i < n; ++i) {
      const uint2 o = s.list[i];
      rank += key_before(__uint_as_float(o.x), static_cast<int>(o.y), k, t) ? 1 : 0;
    }
  }
  __syncthreads();                               // every thread has read the list and its length
  if (tid < n && rank < R) {
    s.list[rank] = make_uint2(__float_as_uint(k), static_cast<uint32_t>(t));
    if (rank == R - 1) s.top[15].x = __float_as_uint(k);
  }
  if (tid == 0) *s.cnt = min(n, R);
  __syncthreads();
  return n >= R ? __uint_as_float(s.top[15].x) : T;
}

__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void dsmem_st_u64(uint32_t addr, uint2 v) {
  asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(addr), "r"(v.x), "r"(v.y) : "memory");
}

// R-th best of the warps' two best entries each (k, j: this thread's best, -inf / 0x7fffffff for none): entries of
// distinct tokens, so a lower bound of the row's R-th best; every warp ranks them for itself.  -inf when fewer are
// finite.  R <= 2 * SW.  One barrier.
__device__ __forceinline__ float first_threshold(const TopList& s, int R, float k, int j) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float k1 = k, k2;
  int j1 = j, j2;
  warp_key_first(k1, j1);
  k2 = (j == j1) ? -INFINITY : k;
  j2 = (j == j1) ? 0x7fffffff : j;
  warp_key_first(k2, j2);
  if (lane == 0) {
    s.pk[2 * warp] = make_uint2(__float_as_uint(k1), static_cast<uint32_t>(j1));
    s.pk[2 * warp + 1] = make_uint2(__float_as_uint(k2), static_cast<uint32_t>(j2));
  }
  __syncthreads();
  const uint2 en = s.pk[lane & (2 * SW - 1)];
  const float mk = __uint_as_float(en.x);
  const int mt = static_cast<int>(en.y);
  int rank = 0;
#pragma unroll
  for (int i = 0; i < 2 * SW; ++i) {
    const float ok = __shfl_sync(0xffffffffu, mk, i);
    const int ot = __shfl_sync(0xffffffffu, mt, i);
    rank += key_before(ok, ot, mk, mt) ? 1 : 0;
  }
  const uint32_t hit = __ballot_sync(0xffffffffu, lane < 2 * SW && rank == R - 1 && mt != 0x7fffffff && mk > -INFINITY);
  return hit ? __shfl_sync(0xffffffffu, mk, __ffs(hit) - 1) : -INFINITY;
}

// The best key of the CTA, after first_threshold and before the buffer is written again; -inf when there is none.
__device__ __forceinline__ float first_best(const TopList& s) {
  float best = -INFINITY;
#pragma unroll
  for (int w = 0; w < SW; ++w) best = fmaxf(best, __uint_as_float(s.pk[2 * w].x));
  return best;
}

// CTA 0: the ordered lists that the CTAs of a row pushed (s.fin, lengths in s.rinfo[].x) -> s.list in order; returns
// their total length.  A barrier separates the result from its readers.
__device__ __forceinline__ int merge_lists(const TopList& s, uint32_t nrank) {
  const int tid = threadIdx.x;
  int nf = 0;
  for (uint32_t r = 0; r < nrank; ++r) nf += static_cast<int>(s.rinfo[r].x);
  const int r_own = tid / kMaxR, i_own = tid - r_own * kMaxR;
  if (r_own < static_cast<int>(nrank) && i_own < static_cast<int>(s.rinfo[r_own].x)) {
    const uint2 en = s.fin[tid];
    int rank = i_own;                                    // the CTAs' lists are in order
    for (uint32_t r = 0; r < nrank; ++r) {
      if (static_cast<int>(r) == r_own) continue;
      const int m = static_cast<int>(s.rinfo[r].x);
#pragma unroll
      for (int i = 0; i < kMaxR; ++i) {
        const uint2 o = s.fin[r * kMaxR + i];
        rank += (i < m && key_before(__uint_as_float(o.x), static_cast<int>(o.y), __uint_as_float(en.x), static_cast<int>(en.y))) ? 1 : 0;
      }
    }
    s.list[rank] = en;                                   // (this CTA's own list has been copied to s.fin)
  }
  __syncthreads();
  return nf;
}

}  // namespace stream
}  // namespace lantern
