// Blackwell tensor path of the latent-neighbour table (Sec. 2.2 / Sec. 4: B_k; App. A.1: the
// codebook): the distance contraction on the fifth-generation tensor cores (tcgen05.mma, bf16 x bf16
// -> float32 accumulators in tensor memory) only selects candidates; the table is exact.
//
//   approximate distance  f(i,j) = |c_i|^2 + g(i,j),  g(i,j) = |c_j|^2 - 2 <c_i, c_j>   (float32)
//   |f - D| <= eps_i for the exact squared distance D, eps_i = ((d+16) 2^-21 [+ 2^-16]) (|c_i|^2 + max_j |c_j|^2)
// (accumulation of the products, the two norms, the final roundings, with a factor of slack).  Rows
// are zero-padded to a multiple of 16 elements (the K extent of one MMA), which changes no inner
// product.  Float32 rows enter as two bfloat16 halves h + l of every element: the query side is laid
// out as [h l h], the candidate side as [h h l], so one contraction of length 3 d gives
// hh + lh + hl; what is missing is below 3 * 2^-18 (1 + 2^-7) |x| |y| per product, which is the 2^-16 term above.
//
// Four kernels per chunk of query tiles (a tile = 128 queries = tensor-memory lanes):
//   knn_t5_kernel<true>    every sampled candidate (one in four, evenly spread): smallest g of every
//                          group of G columns per query, one FMA and one minimum per distance.
//   knn_bound_kernel, knn_t5_kernel<false>
//                          the (k+1)-th smallest of a query's group minima bounds its (k+1)-th
//                          smallest g (the query itself may be among them) whatever the data, so
//                          everything with g <= that + 2 eps is a superset of the neighbours; those
//                          entries are appended to the query's lists, about 4.4 k of them when the
//                          sample is representative.  A list that would overflow all the same is cut
//                          back by its warp.
//   knn_rank_kernel        one CTA per query: cuts the lists down to the k-th smallest g + 2 eps and
//                          ranks the survivors by (exact distance in double precision, index).  Queries whose
//                          survivors are too many (rows closer together than eps) or too few go to knn_rest_kernel.
// Measured on 65536 x 256, k = 200 (5.5 ms; one kernel that streamed from an open threshold, cut lists back
// and ranked behind the contraction took 19.7): per chunk of 18944 queries 0.22 ms sample pass, 0.06 ms bounds,
// 0.75 ms contraction, 0.64 ms ranking; the tensor rate alone would be 0.39 ms per chunk.  The contraction's
// kernel is bound by the issue slots of its selection (nine instructions per distance, 61 % of the slots busy),
// the ranking by issue slots too (widening, double-precision differences, sort).  8192 x 256: 0.42 ms, was 1.59.
// Ranking wants many warps in flight (scattered row reads, long-latency double-precision chains), which is
// why it is a kernel of its own.
//
// knn_t5_kernel: one CTA of 320 threads per (query tile, share of the candidates), candidates in
// tiles of 128 (tensor-memory columns):
//   warp 9     one thread copies operand tiles with cp.async.bulk, two candidate stages in flight: knn_prep_kernel has
//              laid the codebook out once in the K-major core-matrix order the tensor core reads without
//              swizzling (a core matrix = 8 rows x 16 bytes, contiguous), so a tile is one run of bytes;
//   warp 8     one thread issues the MMAs of a tile into one of two 128-column accumulators and
//              commits to the mbarriers that free the stage and publish the accumulator;
//   warps 0-7  two threads per query, 64 columns each (four threads with 32 each: 5.79 ms instead of 5.54 on
//              65536 x 256, k = 200), read their lane of the accumulator with
//              tcgen05.ld and take minima, or append to a list of their own in global memory (no atomics).
// Every wait on an mbarrier is bounded; a wait that runs out raises an abort flag that all roles poll,
// the CTA frees its tensor memory and returns, and the rows of its queries are written as -1.
#pragma once

#include <float.h>

#include "common.cuh"

namespace lantern {

constexpr int kT5Q = 128;           // queries per tile (tensor-memory lanes)
constexpr int kT5C = 128;           // candidates per tile (tensor-memory columns per accumulator)
constexpr int kT5Per = 2;           // threads per query in the selection
constexpr int kT5Cols = kT5C / kT5Per;               // columns of a tile each of them looks at
constexpr int kT5Sel = kT5Per * kT5Q;                // selection threads
constexpr int kT5Mma = kT5Sel / 32;                  // the warp that issues the MMAs; the next one loads
constexpr int kT5Threads = kT5Sel + 64;
constexpr int kT5Sort = 512;        // exact ranking: candidates per query (power of two)
constexpr int kT5MaxK = 320;
constexpr int kT5Items = 148;       // CTAs per chunk (one per SM)
constexpr int kT5MaxSplit = 8;      // shares of the candidates
constexpr int kT5MaxGroups = 1024;  // group minima per query
constexpr float kT5Huge = 1e37f;    // rows with a squared norm from here on (or NaN) never enter the bounds or the lists

struct KnnT5Args {
  // operand tiles of 128 rows in the layout the tensor core reads, [dpad/8 chunks][16 row groups][8 rows][16 bytes]:
  const unsigned char *qm, *cm;     // query side, and candidate side (the sampled rows in the sample pass)
  const float* cn;                  // squared norms of the candidate side's rows, +inf for rows that are none and from kT5Huge on
  const float* nrm;                 // [L] squared norms, nrm[L] = the largest below kT5Huge
  float* minima;                    // [tiles][kT5Q][groups] (sample pass)
  const float* bound;               // [tiles][kT5Q] knn_bound_kernel's result
  unsigned long long* lists;        // [tiles][split][kT5Per][kT5Q][cap]: (bits of g) << 32 | index
  int* counts;                      // [tiles][split][kT5Per][kT5Q] entries; -1: overflow, -9: a wait ran out
  int L, dp, k, cap;                // dp: elements per operand row (a multiple of 16)
  int tile0;                        // first query tile of the chunk
  int split;                        // CTAs per query tile
  int nct;                          // candidate tiles of this pass
  int gshift;                       // log2 of the columns per group minimum (0 .. 5)
  int groups;                       // group minima per query
  float eps1;                       // eps_i = eps1 (|c_i|^2 + max) + eps0
  float eps0;
};

__host__ __device__ constexpr size_t knn_t5_smem(int dp) {
  return static_cast<size_t>(3) * kT5Q * dp * 2                       // query tile, two candidate stages
         + 4 * kT5C * 4                                               // candidate norms, 4 tiles deep
         + kT5Mma * 256 * 4                                           // per-warp histogram of a cut
         + 16 * 8 + 16;                                               // mbarriers, misc
}

// slack for the roundings between the thresholds and g: everything the bound has to cover, in g
__device__ __forceinline__ float t5_margin(const KnnT5Args& a, float nq, float nmax) {
  return 2.f * fmaf(a.eps1, nq + nmax, a.eps0);
}

__device__ __forceinline__ uint64_t t5_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  // shared-memory matrix descriptor, no swizzle: start address, leading (K) and stride (M/N) byte
  // offsets between core matrices, all in units of 16 bytes; descriptor version 1
  return static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4) | (static_cast<uint64_t>((lbo_bytes >> 4) & 0x3FFFu) << 16) |
         (static_cast<uint64_t>((sbo_bytes >> 4) & 0x3FFFu) << 32) | (static_cast<uint64_t>(1) << 46);
}

// bounded wait of one thread on an mbarrier phase that also gives up when another role has raised
// `abort`: the hardware suspends the thread for at most a microsecond per try, so the bound is about a second
__device__ __forceinline__ bool t5_wait(uint32_t mbar, uint32_t parity, volatile int* abort) {
  for (int it = 0; it < (1 << 20); ++it) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(mbar), "r"(parity), "r"(1000u) : "memory");
    if (ok) return true;
    if ((it & 255) == 255 && *abort) return false;
  }
  *abort = 1;
  return false;
}
// the same for a whole warp: lane 0 polls, the result is shared (__shfl_sync orders memory among the lanes)
__device__ __forceinline__ bool t5_wait_warp(uint32_t mbar, uint32_t parity, volatile int* abort) {
  int ok = 1;
  if ((threadIdx.x & 31) == 0) ok = t5_wait(mbar, parity, abort) ? 1 : 0;
  return __shfl_sync(0xffffffffu, ok, 0) != 0;
}
__device__ __forceinline__ void t5_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}

// `bytes` (a multiple of 16) from global to shared memory by bulk copies that complete on `mbar`, which must
// already expect them; pieces of 8 KB, so that one tile is spread over several copy requests.
__device__ __forceinline__ void t5_bulk(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
  const unsigned char* g = static_cast<const unsigned char*>(src);
  for (uint32_t o = 0; o < bytes; o += 8192u) {
    const uint32_t n = min(8192u, bytes - o);
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst + o), "l"(g + o), "r"(n), "r"(mbar) : "memory");
  }
}
__device__ __forceinline__ void t5_expect(uint32_t mbar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void t5_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
               "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                 "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                 "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                 "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
               : "r"(taddr) : "memory");
}

// Digit passes shared by the cuts: narrows (k-th smallest key - kmin) from bit `hi` down by histograms of
// up to 8 bits until its bin holds at most `slack` keys.  count(lo, mask, hi, prefix) fills hist[256]
// (zeroed here); every warp of the caller evaluates the same histogram.  Returns an upper bound of the
// k-th smallest key (the upper edge of its bin, at most kmax).
template <typename SYNC, typename COUNT>
__device__ __forceinline__ uint32_t t5_digit_select(uint32_t kmin, uint32_t kmax, int k, int slack, uint32_t* hist, int tid, int nt,
                                                    SYNC&& sync, COUNT&& count) {
  const int lane = threadIdx.x & 31;
  int hi = 32 - __clz(kmax - kmin);                           // key - kmin < 2^hi
  uint32_t prefix = 0;                                        // (k-th key - kmin) >> hi, known so far
  uint32_t rem = static_cast<uint32_t>(k);
  while (hi > 0) {
    const int lo = hi > 8 ? hi - 8 : 0;
    for (int i = tid; i < 256; i += nt) hist[i] = 0;
    sync();
    count(lo, (1u << (hi - lo)) - 1u, hi, prefix);
    sync();
    uint32_t c8[8], sum = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) { c8[i] = hist[lane * 8 + i]; sum += c8[i]; }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    const uint32_t before = incl - sum;
    const bool mine = before < rem && rem <= incl;            // exactly one lane
    uint32_t bin = 0, nrem = 0, pop = 0;
    if (mine) {
      uint32_t run = before;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (run < rem && rem <= run + c8[i]) { bin = lane * 8 + i; nrem = rem - run; pop = c8[i]; }
        run += c8[i];
      }
    }
    const int owner = (__ffs(__ballot_sync(0xffffffffu, mine)) - 1) & 31;
    bin = __shfl_sync(0xffffffffu, bin, owner);
    rem = __shfl_sync(0xffffffffu, nrem, owner);
    pop = __shfl_sync(0xffffffffu, pop, owner);
    prefix = (prefix << (hi - lo)) | bin;
    hi = lo;
    sync();
    if (pop <= static_cast<uint32_t>(slack)) break;
  }
  // keys whose (key - kmin) >> hi equals prefix: the k-th smallest is among them
  const unsigned long long edge = static_cast<unsigned long long>(kmin) + ((static_cast<unsigned long long>(prefix) + 1ull) << hi) - 1ull;
  return edge < kmax ? static_cast<uint32_t>(edge) : kmax;
}

__device__ __forceinline__ uint32_t t5_entry_key(unsigned long long e) { return float_key(__uint_as_float(static_cast<uint32_t>(e >> 32))); }

// Cut-back of one list of n > k entries by one warp, in place and in order: everything up to an upper
// bound of the k-th smallest g plus `margin` stays.  Returns the number kept; *limit_out is the bound in g.
__device__ __forceinline__ int t5_warp_cut(unsigned long long* lst, int n, int k, float margin, uint32_t* hist, float* limit_out) {
  const int lane = threadIdx.x & 31;
  __syncwarp();                                               // the owner's appends are visible to the warp
  uint32_t kmin = 0xffffffffu, kmax = 0u;
#pragma unroll 4
  for (int i = lane; i < n; i += 32) {
    const uint32_t key = t5_entry_key(lst[i]);
    kmin = min(kmin, key);
    kmax = max(kmax, key);
  }
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  const uint32_t kth = t5_digit_select(kmin, kmax, k, 32, hist, lane, 32, [] { __syncwarp(); },
                                       [&](int lo, uint32_t mask, int hi, uint32_t prefix) {
#pragma unroll 4
    for (int i = lane; i < n; i += 32) {
      const uint32_t rel = t5_entry_key(lst[i]) - kmin;
      if (hi == 32 || (rel >> hi) == prefix) atomicAdd(&hist[(rel >> lo) & mask], 1u);
    }
  });
  const float limit = __fadd_ru(key_float(kth), margin);
  int pos = 0;
  for (int i0 = 0; i0 < n; i0 += 32) {
    const int i = i0 + lane;
    const unsigned long long e = i < n ? lst[i] : 0ull;
    const bool keep = i < n && __uint_as_float(static_cast<uint32_t>(e >> 32)) <= limit;
    const uint32_t m = __ballot_sync(0xffffffffu, keep);      // every lane has read its entry before slots <= i are rewritten
    if (keep) lst[pos + __popc(m & ((1u << lane) - 1u))] = e;
    pos += __popc(m);
    __syncwarp();
  }
  *limit_out = limit;
  return pos;
}

// Upper bound (the edge of a bin of a few) of the (k+1)-th smallest group minimum of every query of the chunk,
// one warp per query; FLT_MAX when fewer are finite.  A kernel of its own: inside the contraction's CTAs, two
// warps per scheduler, the selection took as long as 60 candidate tiles.
__global__ void __launch_bounds__(256) knn_bound_kernel(const float* __restrict__ minima, int queries, int groups, int want, float* __restrict__ bound) {
  __shared__ uint32_t hist_s[8][256];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = blockIdx.x * 8 + warp;
  if (q >= queries) return;
  const float* src = minima + static_cast<size_t>(q) * groups;
  uint32_t* hist = hist_s[warp];
  uint32_t key[kT5MaxGroups / 32];
  uint32_t kmin = 0xffffffffu, kmax = 0u;
  const uint32_t top = float_key(FLT_MAX);
  int finite = 0;
#pragma unroll
  for (int i = 0; i < kT5MaxGroups / 32; ++i) {
    const int m = i * 32 + lane;
    key[i] = m < groups ? float_key(__ldg(src + m)) : 0xffffffffu;
    kmin = min(kmin, key[i]);
    if (key[i] <= top) { kmax = max(kmax, key[i]); ++finite; }
  }
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  finite = __reduce_add_sync(0xffffffffu, finite);
  float v = FLT_MAX;
  if (finite >= want) {
    const uint32_t kth = t5_digit_select(kmin, kmax, want, 8, hist, lane, 32, [] { __syncwarp(); },
                                         [&](int lo, uint32_t mask, int hi, uint32_t prefix) {
#pragma unroll
      for (int i = 0; i < kT5MaxGroups / 32; ++i) {
        const uint32_t rel = key[i] - kmin;
        if (key[i] <= top && (hi == 32 || (rel >> hi) == prefix)) atomicAdd(&hist[(rel >> lo) & mask], 1u);
      }
    });
    v = key_float(kth);
  }
  if (lane == 0) bound[q] = v;
}

template <bool SAMPLE>
__global__ void __launch_bounds__(kT5Threads, 1) knn_t5_kernel(const KnnT5Args a) {
  extern __shared__ __align__(128) unsigned char t5_smem[];
  const int L = a.L, dp = a.dp;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const size_t tile_bytes = static_cast<size_t>(kT5C) * dp * 2;
  unsigned char* As = t5_smem;                                        // [dp/8][16][8][16 B]
  unsigned char* Bs = As + tile_bytes;                                // [2 stages][dp/8][16][8][16 B]
  float* ncs = reinterpret_cast<float*>(Bs + 2 * tile_bytes);         // [4][kT5C] candidate norms
  uint32_t* cut_hist = reinterpret_cast<uint32_t*>(ncs + 4 * kT5C);   // [kT5Mma][256]
  uint64_t* bars = reinterpret_cast<uint64_t*>(cut_hist + kT5Mma * 256);   // full[2] empty[2] tfull[2] tempty[2] afull
  int* misc = reinterpret_cast<int*>(bars + 16);                      // [0] tensor-memory base, [1] abort, [3] the loading thread's last waits

  const uint32_t bar0 = smem_u32(bars);
  auto full = [&](uint32_t s2) { return bar0 + 8u * s2; };
  auto empty = [&](uint32_t s2) { return bar0 + 8u * (2 + s2); };
  auto tfull = [&](uint32_t b) { return bar0 + 8u * (4 + b); };
  auto tempty = [&](uint32_t b) { return bar0 + 8u * (6 + b); };
  const uint32_t afull = bar0 + 8u * 8;
  volatile int* abort = misc + 1;
  if (tid == 0) {
    auto init = [&](uint32_t b, int count) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(b), "r"(count) : "memory"); };
    for (uint32_t s2 = 0; s2 < 2; ++s2) { init(full(s2), 1); init(empty(s2), 1); init(tfull(s2), 1); init(tempty(s2), kT5Sel); }
    init(afull, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    misc[1] = 0;
    misc[3] = 0;
  }
  if (warp == kT5Mma) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(misc)), "r"(2 * kT5C) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tbase = static_cast<uint32_t>(misc[0]);

  // this CTA's query tile (within the chunk) and its share [t0, t1) of the candidate tiles
  const int tile = blockIdx.x / a.split, part = blockIdx.x - tile * a.split;
  const int q0 = (a.tile0 + tile) * kT5Q;
  const int nct = a.nct;
  const int t0 = static_cast<int>(static_cast<long long>(nct) * part / a.split);
  const int t1 = static_cast<int>(static_cast<long long>(nct) * (part + 1) / a.split);
  const float nmax = a.nrm[L];
  bool dead = false;                                // a wait ran out (here or in another role): work is skipped

  if (warp == kT5Mma + 1) {
    // ---------------------------------------------------------------- loads (one thread)
    if (lane == 0) {
      const uint32_t tb = static_cast<uint32_t>(tile_bytes);
      t5_expect(afull, tb);
      t5_bulk(smem_u32(As), a.qm + static_cast<size_t>(a.tile0 + tile) * tile_bytes, tb, afull);
      uint32_t n = 0;
      for (int t = t0; t < t1; ++t, ++n) {
        const uint32_t s2 = n & 1u;
        if (!t5_wait(empty(s2), ((n >> 1) & 1u) ^ 1u, abort)) break;
        t5_expect(full(s2), tb + kT5C * 4u);
        t5_bulk(smem_u32(Bs + s2 * tile_bytes), a.cm + static_cast<size_t>(t) * tile_bytes, tb, full(s2));
        t5_bulk(smem_u32(ncs + (n & 3u) * kT5C), a.cn + static_cast<size_t>(t) * kT5C, kT5C * 4u, full(s2));
      }
      // the CTA may not leave while a copy is on its way into its shared memory
      t5_wait(afull, 0u, abort + 2);
      for (uint32_t back = 1; back <= 2 && back <= n; ++back) t5_wait(full((n - back) & 1u), ((n - back) >> 1) & 1u, abort + 2);
    }
  } else if (warp == kT5Mma) {
    // ---------------------------------------------------------------- tensor-core issue (one thread)
    if (lane == 0) {
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(kT5C >> 3) << 17) |
                             (static_cast<uint32_t>(kT5Q >> 4) << 24);     // f32 += bf16 x bf16, K-major, N, M
      const uint32_t lbo = 16u * 128u, sbo = 128u;
      dead = !t5_wait(afull, 0u, abort);
      for (int t = t0; t < t1; ++t) {
        const uint32_t n = static_cast<uint32_t>(t - t0), s2 = n & 1u, par = (n >> 1) & 1u;
        if (!dead) dead = !t5_wait(full(s2), par, abort);
        if (!dead) dead = !t5_wait(tempty(s2), par ^ 1u, abort);
        if (!dead) {
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t a0 = smem_u32(As), b0 = smem_u32(Bs + s2 * tile_bytes);
          for (int kk = 0; kk < dp / 16; ++kk) {
            const uint64_t da = t5_desc(a0 + kk * 2u * lbo, lbo, sbo);
            const uint64_t db = t5_desc(b0 + kk * 2u * lbo, lbo, sbo);
            const uint32_t acc = kk > 0 ? 1u : 0u;
            asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t"
                         "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                         ::"r"(tbase + s2 * kT5C), "l"(da), "l"(db), "r"(idesc), "r"(acc) : "memory");
          }
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(empty(s2)) : "memory");
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tfull(s2)) : "memory");
        }
      }
    }
  } else {
    // ---------------------------------------------------------------- selection (warps 0-7): two threads per query
    const int q = (warp & 3) * 32 + lane, half = warp >> 2;
    const int qi = q0 + q;
    const float nq = qi < L ? a.nrm[qi] : 0.f;
    const bool active = qi < L && nq < kT5Huge;      // (other rows are ranked without the contraction)
    const float margin = t5_margin(a, nq, nmax);
    float thr = __int_as_float(0x7fffffff);          // NaN: nothing passes (rows without a query)
    if (!SAMPLE && active) thr = fminf(__fadd_ru(a.bound[tile * kT5Q + q], margin), FLT_MAX);
    const size_t seg = static_cast<size_t>((tile * a.split + part) * kT5Per + half) * kT5Q + q;
    float* mins = a.minima + (static_cast<size_t>(tile) * kT5Q + q) * a.groups;
    uint32_t* hist_w = cut_hist + warp * 256;
    const uint32_t base = static_cast<uint32_t>(seg * a.cap * 8);   // (the lists of a chunk take less than 4 GB)
    uint32_t woff = base;                            // byte offset of the next free entry of the own list
    bool ovf = false;
    for (int t = t0; t < t1; ++t) {
      const uint32_t n = static_cast<uint32_t>(t - t0), b = n & 1u;
      if (!dead) dead = !t5_wait_warp(tfull(b), (n >> 1) & 1u, abort);   // warp-uniform
      if (!dead) asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const float* nc = ncs + (n & 3u) * kT5C + half * kT5Cols;
#pragma unroll 1
      for (int c0 = 0; c0 < kT5Cols; c0 += 32) {
        uint32_t r[32];
        if (!dead) {
          t5_ld32(tbase + (static_cast<uint32_t>((warp & 3) * 32) << 16) + b * kT5C + half * kT5Cols + c0, r);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        }
        if (SAMPLE) {
          float v[32];
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = dead ? INFINITY : fmaf(-2.f, __uint_as_float(r[j]), nc[c0 + j]);
          const int gs = a.gshift, G = 1 << gs;
#pragma unroll
          for (int w = 1; w < 32; w *= 2) {
            if (G > w) {
#pragma unroll
              for (int j = 0; j < 32; ++j)
                if (j % (2 * w) == 0) v[j] = fminf(v[j], v[j + w]);
            }
          }
          float* to = mins + ((t * kT5C + half * kT5Cols + c0) >> gs);
          if (G >= 16) {
            to[0] = v[0];
            if (G == 16) to[1] = v[16];
          } else {                                   // four minima and more per 32 columns: 16-byte stores
#pragma unroll
            for (int w = 1; w < 16; w *= 2) {
              if (G == w) {
#pragma unroll
                for (int j = 0; j < 32 / w; j += 4)
                  *reinterpret_cast<float4*>(to + j) = make_float4(v[j * w], v[(j + 1) * w], v[(j + 2) * w], v[(j + 3) * w]);
              }
            }
          }
        } else if (!dead && !ovf) {
          const int cbase = t * kT5C + half * kT5Cols + c0;
          // per candidate: one FMA, one compare, and a store and pointer step that are predicated in the
          // instruction stream (a branch here would diverge on a fifth of the candidates)
#pragma unroll
          for (int j4 = 0; j4 < 32; j4 += 4) {
            const float4 n4 = *reinterpret_cast<const float4*>(nc + c0 + j4);
            const float nn[4] = {n4.x, n4.y, n4.z, n4.w};
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) {
              const float g = fmaf(-2.f, __uint_as_float(r[j4 + jj]), nn[jj]);
              asm volatile("{\n\t.reg .pred p;\n\tsetp.le.f32 p, %1, %2;\n\t"
                           ".reg .u64 a;\n\tcvt.u64.u32 a, %0;\n\tadd.u64 a, %4, a;\n\t"
                           "@p st.global.v2.b32 [a], {%3, %1};\n\t"
                           "@p add.u32 %0, %0, 8;\n\t}"
                           : "+r"(woff) : "f"(g), "f"(thr), "r"(cbase + j4 + jj), "l"(a.lists) : "memory");
            }
          }
        }
      }
      if (!dead) {
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        t5_arrive(tempty(b));
      }
      if (!SAMPLE) {
        // a list that could overflow during the next tile is cut back by its warp
        uint32_t m = __ballot_sync(0xffffffffu, !ovf && !dead && static_cast<int>((woff - base) >> 3) > a.cap - kT5Cols);
        while (m) {
          const int src = __ffs(m) - 1;
          m &= m - 1;
          const int cnt = __shfl_sync(0xffffffffu, static_cast<int>((woff - base) >> 3), src);
          const float mg = __shfl_sync(0xffffffffu, margin, src);
          unsigned long long* lq = a.lists + (static_cast<size_t>((tile * a.split + part) * kT5Per + half) * kT5Q + (warp & 3) * 32 + src) * a.cap;
          float limit;
          const int kept = t5_warp_cut(lq, cnt, a.k + 1, mg, hist_w, &limit);
          if (lane == src) {
            woff = base + static_cast<uint32_t>(kept) * 8u;
            thr = fminf(thr, limit);
            if (kept > a.cap - kT5Cols) ovf = true;              // too many rows within the error margin
          }
        }
      }
    }
    if (!SAMPLE) a.counts[seg] = dead ? -9 : (ovf || !active ? -1 : static_cast<int>((woff - base) >> 3));
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == kT5Mma) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(2 * kT5C) : "memory");
}

// Squared norms (float32) and the largest of those below kT5Huge, and the operand tiles (the layout is at KnnT5Args):
// [h l h] and [h h l] of float32 elements (each part d elements) on the query and the candidate side, bfloat16
// rows as they are on both, zero beyond.  One warp per row of a tile; rows from `tiles` * 128 on are those of the
// sample, row i of it being codebook row (i * step) >> 32.  The eight warps of a CTA write one row group, 128
// contiguous bytes per chunk.
struct KnnPrepArgs {
  const void* cb;
  int L, d, dp, rows, sampled;      // tile rows of the candidate side, of the sample (multiples of 128; 0: no sample tiles)
  unsigned long long step;
  float *nrm, *cn, *sn;             // nrm[L + 1]: non-zero when an element is not +0 and not of ordinary size (bfloat16 rows)
  unsigned char *qm, *cm, *sm;      // cm == qm for bfloat16 rows
};
template <typename T>
__global__ void __launch_bounds__(256) knn_prep_kernel(const KnnPrepArgs a) {
  const int out = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  const bool sample = out >= a.rows;
  const int tr = sample ? out - a.rows : out;                  // row among the tiles of its side
  const int row = sample ? static_cast<int>((static_cast<unsigned long long>(tr) * a.step) >> 32) : tr;
  const bool in = row < a.L;
  const int d = a.d, dp = a.dp;
  const T* src = static_cast<const T*>(a.cb) + static_cast<long long>(in ? row : 0) * d;
  float s = 0.f;
  bool odd = false;                                            // -0, below 2^-60, infinite or NaN
  for (int t = lane; t < d; t += 32) {
    const float v = static_cast<float>(src[t]);
    s = fmaf(v, v, s);
    odd |= !(fabsf(v) >= 8.673617379884035e-19f && fabsf(v) <= FLT_MAX) && __float_as_uint(v) != 0u;
  }
  s = warp_sum(s);
  odd = __any_sync(0xffffffffu, odd);
  if (lane == 0) {
    if (odd && !sample && in) a.nrm[a.L + 1] = 1.f;
    // (a row whose norm the error bound does not cover is no candidate: a query that needs it finds too few others)
    (sample ? a.sn : a.cn)[tr] = in && s < kT5Huge ? s : INFINITY;
    if (!sample && in) {
      a.nrm[row] = s;
      unsigned int* top = reinterpret_cast<unsigned int*>(a.nrm + a.L);      // s >= 0: bit order = value order
      if (s < kT5Huge && __float_as_uint(s) > __ldcg(top)) atomicMax(top, __float_as_uint(s));
    }
  }
  const size_t base = static_cast<size_t>(tr >> 7) * (static_cast<size_t>(dp) * 256) + static_cast<size_t>((tr & 127) >> 3) * 128 + (tr & 7) * 16;
  for (int c = lane; c < dp / 8; c += 32) {
    union { __nv_bfloat16 h[8]; uint4 v; } x, y;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int t = c * 8 + e;
      x.h[e] = y.h[e] = __float2bfloat16_rn(0.f);
      if (sizeof(T) == 2) {
        if (in && t < d) x.h[e] = __float2bfloat16_rn(static_cast<float>(src[t]));
      } else if (in && t < 3 * d) {
        const int part = t / d;
        const float v = static_cast<float>(src[t - part * d]);
        const __nv_bfloat16 h = __float2bfloat16_rn(v), l = __float2bfloat16_rn(v - __bfloat162float(h));
        x.h[e] = part == 1 ? l : h;
        y.h[e] = part == 2 ? l : h;
      }
    }
    const size_t at = base + static_cast<size_t>(c) * 2048;
    if (sizeof(T) == 2) {
      *reinterpret_cast<uint4*>((sample ? a.sm : a.qm) + at) = x.v;
    } else {
      if (!sample) *reinterpret_cast<uint4*>(a.qm + at) = x.v;
      *reinterpret_cast<uint4*>((sample ? a.sm : a.cm) + at) = y.v;
    }
  }
}

// ------------------------------------------------------------------------------------ exact ranking
struct KnnRankArgs {
  const void* cb;
  const float* nrm;
  const unsigned long long* lists;
  const int* counts;
  int L, d, k, cap, split;
  int q0;                           // first query of the chunk
  int lanes;                        // lanes that share one candidate's distance (power of two); 0: rows read element by element
  float eps1, eps0;
  int *rest, *n_rest;               // queries left to the brute-force kernel, and their number
  int32_t* nbr_idx;
  float* nbr_dist;
};
constexpr int kRankThreads = 128;
__host__ __device__ constexpr size_t knn_rank_smem(int d) {
  return kT5Sort * (8 + 8 + 4) + 256 * 4 + static_cast<size_t>((d + 7) / 8 * 8) * 8 + 16;
}

// Eight elements to double.  For normal bfloat16 numbers the double's high word is the sign, the exponent rebiased by
// 1023 - 127 and the 7 mantissa bits: integer operations instead of the converting instruction's quarter rate.
// The same operations turn +0 into 2^-127, which changes no difference with a number of at least 2^-60 in
// magnitude and none between zeros; codebooks with anything else (knn_prep_kernel looks) take the instruction (PLAIN).
__device__ __forceinline__ double bf16_high_to_double(uint32_t w) {          // the upper 16 bits
  return __hiloint2double((static_cast<int>(w) >> 3 & static_cast<int>(0x8fffe000u)) + (896 << 20), 0);
}
template <bool PLAIN>
__device__ __forceinline__ void widen8(const __nv_bfloat16* p, double (&x)[8]) {
  const uint4 v = __ldg(reinterpret_cast<const uint4*>(p));
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    x[2 * i] = PLAIN ? static_cast<double>(__uint_as_float(w[i] << 16)) : bf16_high_to_double(w[i] << 16);
    x[2 * i + 1] = PLAIN ? static_cast<double>(__uint_as_float(w[i] & 0xffff0000u)) : bf16_high_to_double(w[i]);
  }
}
template <bool PLAIN>
__device__ __forceinline__ void widen8(const float* p, double (&x)[8]) {
  const float4 v = __ldg(reinterpret_cast<const float4*>(p)), w = __ldg(reinterpret_cast<const float4*>(p) + 1);
  x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w; x[4] = w.x; x[5] = w.y; x[6] = w.z; x[7] = w.w;
}

// Exact squared distances between the query row `qd` (pair e of chunk c at pair e * (d / 8) + c) and the n candidates of
// `st`: G lanes per candidate, lane g of them sums the elements [8 c, 8 c + 8), c = g (mod G).
template <typename T, bool PLAIN>
__device__ __forceinline__ void exact_block(const T* __restrict__ cb, int d, int G, const double* qd, const unsigned long long* st, int n,
                                            unsigned long long* sortd, int* sorti) {
  const int tid = threadIdx.x, g = tid & (G - 1), per = kRankThreads / G, nch = d >> 3;
  for (int i0 = 0; i0 < n; i0 += per) {
    const int i = i0 + tid / G;
    const int j = i < n ? static_cast<int>(st[i] & 0xffffffffu) : 0;
    const T* row = cb + static_cast<long long>(j) * d;
    double s = 0.0;
#pragma unroll 4
    for (int c = g; c < nch; c += G) {
      double x[8];
      widen8<PLAIN>(row + c * 8, x);
      const double2* qp = reinterpret_cast<const double2*>(qd) + c;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const double2 qv = qp[e * nch];
        const double d0 = qv.x - x[2 * e], d1 = qv.y - x[2 * e + 1];
        s = fma(d0, d0, s);
        s = fma(d1, d1, s);
      }
    }
    for (int o = 1; o < G; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (g == 0 && i < n) { sorti[i] = j; sortd[i] = static_cast<unsigned long long>(__double_as_longlong(s)); }
  }
}

// One CTA of 128 threads per query, up to 16 of them per SM: every step is short, and what bounds it is
// the latency of scattered row reads (L2) and of the double-precision chains, so warps in flight count.
// A candidate's distance is shared by up to 8 lanes, 8 consecutive elements (one or two 16-byte loads) each, so
// that a warp reads whole 128-byte lines.
template <typename T>
__global__ void __launch_bounds__(kRankThreads) knn_rank_kernel(const KnnRankArgs a) {
  extern __shared__ __align__(16) unsigned char rank_smem[];
  unsigned long long* st = reinterpret_cast<unsigned long long*>(rank_smem);     // [kT5Sort] survivors
  unsigned long long* sortd = st + kT5Sort;                                      // [kT5Sort] bits of doubles >= 0
  double* qd = reinterpret_cast<double*>(sortd + kT5Sort);                       // [d] the query row
  int* sorti = reinterpret_cast<int*>(qd + (a.d + 7) / 8 * 8);                   // [kT5Sort]
  uint32_t* hist = reinterpret_cast<uint32_t*>(sorti + kT5Sort);                 // [256]
  int* misc = reinterpret_cast<int*>(hist + 256);                                // [0] survivors
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const T* cb = static_cast<const T*>(a.cb);
  const int ql = blockIdx.x, qi = a.q0 + ql, k = a.k, d = a.d;
  const int nseg = a.split * kT5Per;
  int32_t* out_i = a.nbr_idx + static_cast<long long>(qi) * k;
  float* out_d = a.nbr_dist ? a.nbr_dist + static_cast<long long>(qi) * k : nullptr;
  const size_t seg0 = static_cast<size_t>(ql / kT5Q) * nseg * kT5Q + ql % kT5Q;      // segment s: + s * kT5Q
  const float nq = a.nrm[qi], nmax = a.nrm[a.L];
  const bool nrm_odd = a.nrm[a.L + 1] != 0.f;
  bool lost = false, whole = nq < kT5Huge && nmax < 1e35f;
  for (int s = 0; s < nseg; ++s) {
    const int c = a.counts[seg0 + static_cast<size_t>(s) * kT5Q];
    lost |= c == -9;
    whole &= c >= 0;
  }
  if (lost) {                                        // a wait of the contraction ran out
    for (int r = tid; r < k; r += kRankThreads) { out_i[r] = -1; if (out_d) out_d[r] = 0.f; }
    return;
  }
  // the query row in double precision; pair e of chunk c (elements 8 c + 2 e, + 1) at pair e * (d / 8) + c, so that the
  // lanes of one candidate read consecutive 16-byte words
  if (a.lanes > 0)
    for (int t = tid; t < d; t += kRankThreads)
      qd[(((t & 7) >> 1) * (d >> 3) + (t >> 3)) * 2 + (t & 1)] =
          (sizeof(T) == 4 || nrm_odd) ? static_cast<double>(static_cast<float>(cb[static_cast<long long>(qi) * d + t]))
                                      : bf16_high_to_double(__float_as_uint(static_cast<float>(cb[static_cast<long long>(qi) * d + t])));
  if (tid == 0) misc[0] = 0;
  // fn(entry, whether there is one) for every list entry but the query itself, by whole warps
  auto for_each = [&](auto&& fn) {
    for (int s = 0; s < nseg; ++s) {
      const size_t seg = seg0 + static_cast<size_t>(s) * kT5Q;
      const unsigned long long* lst = a.lists + seg * a.cap;
      const int n = a.counts[seg];
      for (int i0 = warp * 32; i0 < n; i0 += kRankThreads) {
        const int i = i0 + lane;
        const unsigned long long e = i < n ? lst[i] : 0ull;
        fn(e, i < n && static_cast<int>(e & 0xffffffffu) != qi);
      }
    }
  };
  int n = 0;
  if (whole) {
    uint32_t kmin = 0xffffffffu, kmax = 0u;
    int cnt = 0;
    for_each([&](unsigned long long e, bool in) {
      const uint32_t key = t5_entry_key(e);
      if (in) {
        kmin = min(kmin, key);
        kmax = max(kmax, key);
        ++cnt;
      }
    });
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0) { hist[warp] = kmin; hist[4 + warp] = kmax; hist[8 + warp] = static_cast<uint32_t>(cnt); }
    __syncthreads();
    kmin = min(min(hist[0], hist[1]), min(hist[2], hist[3]));
    kmax = max(max(hist[4], hist[5]), max(hist[6], hist[7]));
    cnt = static_cast<int>(hist[8] + hist[9] + hist[10] + hist[11]);
    __syncthreads();
    whole = cnt >= k;
    if (whole) {
      uint32_t kth = kmax;
      if (cnt > k)
        kth = t5_digit_select(kmin, kmax, k, 2, hist, tid, kRankThreads, [] { __syncthreads(); },
                              [&](int lo, uint32_t mask, int hi, uint32_t prefix) {
          for_each([&](unsigned long long e, bool in) {
            const uint32_t rel = t5_entry_key(e) - kmin;
            if (in && (hi == 32 || (rel >> hi) == prefix)) atomicAdd(&hist[(rel >> lo) & mask], 1u);
          });
        });
      const float limit = __fadd_ru(key_float(kth), 2.f * fmaf(a.eps1, nq + nmax, a.eps0));
      for_each([&](unsigned long long e, bool in) {
        const bool keep = in && __uint_as_float(static_cast<uint32_t>(e >> 32)) <= limit;
        const uint32_t m = __ballot_sync(0xffffffffu, keep);
        if (m == 0u) return;
        int pos = 0;
        if (lane == 0) pos = atomicAdd(&misc[0], __popc(m));
        pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(m & ((1u << lane) - 1u));
        if (keep && pos < kT5Sort) st[pos] = e;
      });
      __syncthreads();
      n = misc[0];
      whole = n <= kT5Sort;
    }
  } else {
    __syncthreads();
  }
  if (!whole) {                                      // too few or too many rows under the bound: crowded rows, huge norms
    if (tid == 0) a.rest[atomicAdd(a.n_rest, 1)] = qi;
    return;
  }
  int p2 = 32;
  while (p2 < n) p2 *= 2;
  if (a.lanes > 0) {
    if (sizeof(T) == 4 || nrm_odd) exact_block<T, true>(cb, d, a.lanes, qd, st, n, sortd, sorti);
    else exact_block<T, false>(cb, d, a.lanes, qd, st, n, sortd, sorti);
  } else {
    for (int i = tid; i < n; i += kRankThreads) {
      const int j = static_cast<int>(st[i] & 0xffffffffu);
      sorti[i] = j;
      sortd[i] = static_cast<unsigned long long>(__double_as_longlong(exact_dist<T>(cb, d, qi, j)));
    }
  }
  for (int i = n + tid; i < p2; i += kRankThreads) { sorti[i] = 0x7fffffff; sortd[i] = 0x7ff0000000000000ull; }
  __syncthreads();
  // ascending bitonic sort of (distance, index): non-negative doubles order like their bit patterns
  for (int size = 2; size <= p2; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = tid; i < (p2 >> 1); i += kRankThreads) {
        const int lo = 2 * i - (i & (stride - 1)), hi = lo + stride;
        const bool up = (lo & size) == 0;
        const unsigned long long dx = sortd[lo], dy = sortd[hi];
        const int ix = sorti[lo], iy = sorti[hi];
        const bool gt = dx > dy || (dx == dy && ix > iy);
        if (gt == up) { sortd[lo] = dy; sortd[hi] = dx; sorti[lo] = iy; sorti[hi] = ix; }
      }
      __syncthreads();
    }
  }
  for (int r = tid; r < k; r += kRankThreads) {
    out_i[r] = sorti[r];
    if (out_d) out_d[r] = static_cast<float>(__longlong_as_double(static_cast<long long>(sortd[r])));
  }
}

}  // namespace lantern
