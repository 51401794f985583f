// Rows that are truncated to their top-k entries (App. B "Models"), vocabularies beyond the 16384 tokens whose rows the
// kernels of verify_sparse.cuh hold in shared memory: the row is never held on chip.  A CTA of 512 threads
//   1. reads a sample (a pair of 16-byte vectors of every group of 16, 8192 entries at most), whose histogram gives
//      a value that a little more than the k largest entries of the whole row reach;
//   2. streams the row once and appends what reaches it to a list in shared memory;
//   3. finds the exact k-th largest among those (histogram of max - z, exact ranking inside the
//      located bin) and keeps what is not below it.
// A row whose sample misled (too few or too many entries reach the value) or whose ties do not fit the fixed buffers is
// left to the dense kernel.  Bound: HBM and the chain of short phases behind the row.  65536 float32 logits with
// guidance, k = 2000: 240 nodes 98 us and 144 drafter rows 41 us (the dense kernels, eight CTAs per row: 251 and 126).
// Narrower rows stay on the staged kernels: 480 nodes of 16384 logits, k = 1000, take 65 us here (69 us with the row in
// registers in place of the sample), 48 us there, where all of a row's loads are in flight at once.
#pragma once

#include "toplist.cuh"
#include "verify_sparse.cuh"

namespace lantern {
namespace wide {

using sparse::block_reduce2;
using sparse::Ctx;
using sparse::kCand;
using sparse::kMisc;
using sparse::ST;
using sparse::SW;
constexpr int kMaxV = 131072;      // widest row
constexpr int kMaxTopK = 2048;     // largest top-k routed here
constexpr int kSample = 8192;      // entries of the sample at most
constexpr int kRaw = 4096;         // entries that may reach the sampled value (rows of up to that many skip the sample)

// list entries per side for top-k of k: room for ties at the threshold
__host__ __device__ constexpr int list_cap(int k) { return (k + 256 + 31) / 32 * 32; }
__host__ __device__ constexpr int bitmap_words(int V) { return (V + 127) / 128 * 4; }
// floats of the region that holds the sample, the entries above the sampled value and then the union arrays
__host__ __device__ constexpr int region_floats(int cap) { return 4 * cap > 2 * kRaw ? 4 * cap : 2 * kRaw; }
__host__ __device__ constexpr int bins_words(int V) { return bitmap_words(V) > kBins ? bitmap_words(V) : kBins; }   // histogram, then ranks
static_assert(kSample <= 2 * kRaw, "the sample shares the region");

struct Smem {
  float* rz;         // [kRaw]       entries that reach the sampled value: pre-softmax value ([kSample] with rt: the sample)
  int* rt;           // [kRaw]       ... and token
  uint32_t* bins;    // [kBins]
  float* cand;       // [kCand]
  uint32_t* wtot;    // [SW]
  int* misc;         // [kMisc]
};

// The smallest bin whose cumulative count reaches `need` (>= 1): misc[0] = bin, misc[1] = rank inside it, misc[2] = its
// count.  Every thread calls; a barrier must separate the last count from the call and the call from the read.
__device__ __forceinline__ void locate_bin(const Smem& s, uint32_t need) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  static_assert(kBins == 4 * ST, "four bins per thread");
  const uint4 b4 = *reinterpret_cast<const uint4*>(s.bins + 4 * tid);
  const uint32_t c0 = b4.x, c1 = c0 + b4.y, c2 = c1 + b4.z, c3 = c2 + b4.w;
  uint32_t incl = c3;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) s.wtot[warp] = incl;
  __syncthreads();
  uint32_t wt = lane < SW ? s.wtot[lane] : 0u, wincl = wt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, wincl, o);
    if (lane >= o) wincl += t;
  }
  const uint32_t before = __shfl_sync(0xffffffffu, wincl - wt, warp) + incl - c3;
  const uint32_t lo4[4] = {before, before + c0, before + c1, before + c2};
  const uint32_t cn4[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (lo4[i] < need && need <= lo4[i] + cn4[i]) {
      s.misc[0] = 4 * tid + i;
      s.misc[1] = static_cast<int>(need - lo4[i]);
      s.misc[2] = static_cast<int>(cn4[i]);
    }
  }
}

// Room for `cnt` entries of this lane in a list whose length is *len: one atomic per warp.
__device__ __forceinline__ int reserve(int cnt, int* len) {
  const int lane = threadIdx.x & 31;
  int incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  int base = 0;
  if (lane == 31) base = atomicAdd(len, incl);
  return __shfl_sync(0xffffffffu, base, 31) + incl - cnt;
}

// How many of the sample's largest entries the value to reach is taken from, when the sample holds the share f of
// the row: the expected number of the k largest entries in it and five and a half standard deviations.
__device__ __forceinline__ int sample_rank(int kth, float f) {
  const float kf = static_cast<float>(kth) * f;
  return static_cast<int>(kf + 5.5f * sqrtf(kf)) + 5;
}
// the value below the located bin, from which on everything up to the bin's far edge is taken
__device__ __forceinline__ float bin_floor(float mx, int bin) {
  return bin >= 0 && bin < kBins - 1 ? __fsub_rd(mx, __uint_as_float(bin_hi_bits(bin))) : -INFINITY;
}

// misc[3] = the krem-th largest of the nb candidates: the value v with #(> v) < krem <= #(>= v); eight lanes share the
// comparisons of one candidate
__device__ __forceinline__ void rank_candidates(const Smem& s, int nb, int krem) {
  const int tid = threadIdx.x;
  const int nc8 = (nb + (ST / 8) - 1) / (ST / 8) * (ST / 8);
  for (int i = tid >> 3; i < nc8; i += ST / 8) {
    const float v = i < nb ? s.cand[i] : 0.f;
    int gt = 0, ge = 0;
    for (int t = tid & 7; t < nb; t += 8) {
      const float w = s.cand[t];
      gt += (w > v);
      ge += (w >= v);
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
      gt += __shfl_xor_sync(0xffffffffu, gt, o);
      ge += __shfl_xor_sync(0xffffffffu, ge, o);
    }
    if (i < nb && (tid & 7) == 0 && gt < krem && krem <= ge) reinterpret_cast<float*>(s.misc)[3] = v;
  }
}

// theta = the exact kth-th largest value of the list of n_raw entries (mx: its maximum); false when too many share
// its bin.  The bins are clear.  -inf when no entry has to go.
__device__ __forceinline__ bool list_theta(const Smem& s, int n_raw, float mx, int kth, float& theta) {
  const int tid = threadIdx.x;
  theta = -INFINITY;
  if (n_raw <= kth) return true;
  for (int i = tid; i < n_raw; i += ST) atomicAdd(&s.bins[dist_bin(mx, s.rz[i])], 1u);
  __syncthreads();
  locate_bin(s, static_cast<uint32_t>(kth));
  __syncthreads();
  const int bstar = s.misc[0], krem = s.misc[1], nb = s.misc[2];
  if (nb > kCand) return false;
  const uint32_t hi_bits = bin_hi_bits(bstar), lo_bits = bin_lo_bits(bstar);
  for (int i = tid; i < n_raw; i += ST) {
    const uint32_t d = __float_as_uint(mx - s.rz[i]);
    if (d >= lo_bits && d <= hi_bits) s.cand[atomicAdd(&s.misc[9], 1)] = s.rz[i];
  }
  __syncthreads();
  rank_candidates(s, nb, krem);
  __syncthreads();
  theta = reinterpret_cast<const float*>(s.misc)[3];
  return true;
}

// One row: the entries that reach the sampled value -> (rz, rt), n_raw of them in no particular order; mx = the
// row's maximum, theta = its exact kth-th largest value (-inf: every entry counts).  False when the row does not
// fit: the same answer in every thread.
template <typename IO>
__device__ __forceinline__ bool stream_topk(Ctx& c, const Smem& s, const IO& io, const stream::Geo& ge, int kth, int& n_raw,
                                            float& mx, float& theta) {
  constexpr int VN = IO::VN;
  constexpr int U = IO::kGuided ? 8 / VN : 16 / VN;      // vectors per thread and operand in flight
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float t0 = -INFINITY;
  for (int i = tid; i < kBins; i += ST) s.bins[i] = 0;
  if (tid == 0) { s.misc[8] = 0; s.misc[9] = 0; s.misc[0] = -1; }      // list and candidate counters, no bin located
  // ---- sample: one pair of vectors of every group, at a place that moves from group to group
  if (ge.ahi - ge.alo > kRaw) {
    int gshift = 4;                                      // vectors per group: 16 and up
    while (((ge.vi1 - ge.vi0) >> gshift) * 2 * VN > kSample) ++gshift;
    const int ns = ((ge.vi1 - ge.vi0) >> gshift) * 2;    // sampled vectors
    float m2[2] = {-INFINITY, -INFINITY};
    for (int i = tid; i < ns; i += ST) {
      const int g = i >> 1;
      const int vv = ge.vi0 + (g << gshift) + 2 * ((g * 5 + (g >> 3)) & ((1 << (gshift - 1)) - 1)) + (i & 1);
      uint4 rc, ru;
      io.load(vv, rc, ru);
      float z[VN];
      io.z(rc, ru, z);
#pragma unroll
      for (int e = 0; e < VN; ++e) {
        m2[0] = fmaxf(m2[0], z[e]);
        s.rz[i * VN + e] = z[e];
      }
    }
    block_reduce2<true>(c, m2);                          // (its barrier also publishes the cleared bins)
    if (m2[0] > -INFINITY) {
      for (int i = tid; i < ns; i += ST) {
#pragma unroll
        for (int e = 0; e < VN; ++e) atomicAdd(&s.bins[dist_bin(m2[0], s.rz[i * VN + e])], 1u);
      }
      __syncthreads();
      const int r = sample_rank(kth, 2.f / static_cast<float>(1 << gshift));
      if (r <= ns * VN) {
        locate_bin(s, static_cast<uint32_t>(r));
        __syncthreads();
        t0 = bin_floor(m2[0], s.misc[0]);
      }
    }
    __syncthreads();                                     // the sample's place is free, misc[0] has been read
    for (int i = tid; i < kBins; i += ST) s.bins[i] = 0;
  }
  __syncthreads();
  // ---- the row, once
  for (int base = warp * 32 * U; base < ge.nvec; base += SW * 32 * U) {
    uint4 rc[U], ru[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int vv = base + 32 * u + lane;
      if (vv >= ge.vi0 && vv < ge.vi1) io.load(vv, rc[u], ru[u]);
    }
    float z[U][VN];
    uint32_t mask = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int vv = base + 32 * u + lane;
      if (vv >= ge.vi0 && vv < ge.vi1) {
        io.z(rc[u], ru[u], z[u]);
      } else {                                           // ragged first / last vector, or beyond the row
#pragma unroll
        for (int e = 0; e < VN; ++e) {
          const int t = ge.j0 + vv * VN + e;
          z[u][e] = (vv < ge.nvec && t >= ge.alo && t < ge.ahi) ? io.z_at(t) : -INFINITY;
        }
      }
#pragma unroll
      for (int e = 0; e < VN; ++e)
        if (z[u][e] >= t0 && z[u][e] > -INFINITY) mask |= 1u << (u * VN + e);
    }
    if (!__any_sync(0xffffffffu, mask != 0u)) continue;
    int pos = reserve(__popc(mask), &s.misc[8]);
#pragma unroll
    for (int u = 0; u < U; ++u) {
#pragma unroll
      for (int e = 0; e < VN; ++e) {
        if ((mask >> (u * VN + e)) & 1u) {
          if (pos < kRaw) { s.rz[pos] = z[u][e]; s.rt[pos] = ge.j0 + (base + 32 * u + lane) * VN + e; }
          ++pos;
        }
      }
    }
  }
  __syncthreads();
  n_raw = s.misc[8];
  if (n_raw > kRaw || n_raw == 0 || (n_raw < kth && t0 > -INFINITY)) return false;
  float m2[2] = {-INFINITY, -INFINITY};
  for (int i = tid; i < n_raw; i += ST) m2[0] = fmaxf(m2[0], s.rz[i]);
  block_reduce2<true>(c, m2);
  mx = m2[0];
  return list_theta(s, n_raw, mx, kth, theta);
}

// Geometry of a row's allowed tokens for the streaming loads (one CTA per row)
template <int VN>
__device__ __forceinline__ stream::Geo row_geo(int alo, int ahi) {
  stream::Geo ge;
  ge.alo = alo; ge.ahi = ahi;
  ge.j0 = alo / VN * VN;
  ge.nvec = (ahi - ge.j0 + VN - 1) / VN;
  ge.vi0 = alo > ge.j0 ? 1 : 0;
  ge.vi1 = (ge.j0 + ge.nvec * VN > ahi) ? ge.nvec - 1 : ge.nvec;
  if (ge.vi1 < ge.vi0) ge.vi1 = ge.vi0;
  ge.vw = ge.nvec;
  return ge;
}

}  // namespace wide
}  // namespace lantern
