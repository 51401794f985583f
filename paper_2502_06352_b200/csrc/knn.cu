// Latent-neighbour table (Sec. 2.2 / Sec. 4: B_k = k nearest codebook entries; App. A.1:
// codebook C = {c_1..c_L}, c_i in R^d).  Exact squared-Euclidean k-NN of every row, ordered
// by (distance, index), self excluded.
//
// Exact brute-force kernel.  A CTA owns a tile of QT query rows and streams over all L
// candidate rows; distances are accumulated in double precision (sum of squared differences,
// so duplicate rows give distance exactly 0 and equal distances to third rows).  Selection is
// streaming: per query a float32 threshold tau (the k-th smallest rounded distance seen so
// far) filters candidates into a shared-memory buffer; when the buffer fills it is sorted and
// cut back to the entries <= the new tau (rounding to float32 is monotone, so nothing that can
// belong to the exact top k is ever dropped).  The survivors are re-ranked by their double
// distances.  If ties at tau overflow the buffer the query falls back to k rounds of an exact
// arg-min over all candidates.
#include <math.h>

#include "common.cuh"

namespace lantern {

constexpr int kKnnThreads = 256;
constexpr int kDC = 32;             // embedding dims staged per step

struct KnnArgs {
  const void* cb;
  int L, d, k, QT, CAP, q_double;
  int f32acc;        // filter distances accumulated in float32 with an error margin (small d)
  float margin;      // 1 + 3 (d + 2) 2^-24: the filter keeps everything within this factor of tau ...
  float slack;       // ... and this much more: the rounding of sums below the normal range
  int32_t* nbr_idx;
  float* nbr_dist;
  const int *queries, *n_queries;   // LISTED: the query rows, in any order, and their number
};

template <typename T> __device__ __forceinline__ float widen(T x);
template <> __device__ __forceinline__ float widen<float>(float x) { return x; }
template <> __device__ __forceinline__ float widen<__nv_bfloat16>(__nv_bfloat16 x) { return __bfloat162float(x); }

// ascending bitonic sort of n (power of two) (dist, idx) pairs
__device__ __forceinline__ void bitonic_pair(double* dv, int* iv, int n) {
  for (int size = 2; size <= n; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = threadIdx.x; i < (n >> 1); i += kKnnThreads) {
        int lo = 2 * i - (i & (stride - 1));
        int hi = lo + stride;
        bool up = (lo & size) == 0;
        double dx = dv[lo], dy = dv[hi];
        int ix = iv[lo], iy = iv[hi];
        bool gt = dx > dy || (dx == dy && ix > iy);
        if (gt == up) { dv[lo] = dy; dv[hi] = dx; iv[lo] = iy; iv[hi] = ix; }
      }
      __syncthreads();
    }
  }
}

// Cut-back of one query's candidate buffer without sorting it.  Entries are 64-bit words whose
// upper half is a monotone 32-bit key of the filter distance.  A most-significant-digit radix
// select (4 passes of 8 bits, shared-memory histogram) finds the k-th smallest key; `limit_of`
// turns it into the largest key that may stay (k-th key plus the caller's error margin); the
// entries up to that limit are compacted through `tmp` (order is irrelevant: the final ranking
// sorts).  Returns the number kept; *kth_key_out receives the k-th smallest key.  n >= k.
template <typename F>
__device__ __forceinline__ int radix_cut(unsigned long long* bq, int n, int k, unsigned long long* tmp, uint32_t* hist,
                                         int* sel, F&& limit_of, uint32_t* limit_out) {
  const int tid = threadIdx.x, lane = tid & 31;
  uint32_t prefix = 0;
  int rem = k;
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 24 - 8 * pass;
    for (int i = tid; i < 256; i += kKnnThreads) hist[i] = 0;
    __syncthreads();
    for (int i = tid; i < n; i += kKnnThreads) {
      const uint32_t key = static_cast<uint32_t>(bq[i] >> 32);
      if (pass == 0 || (key >> (shift + 8)) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (tid < 32) {
      uint32_t c8[8], s = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) { c8[i] = hist[lane * 8 + i]; s += c8[i]; }
      uint32_t incl = s;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
      }
      const uint32_t before = incl - s;
      if (before < static_cast<uint32_t>(rem) && static_cast<uint32_t>(rem) <= incl) {     // exactly one lane
        uint32_t run = before;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          if (run < static_cast<uint32_t>(rem) && static_cast<uint32_t>(rem) <= run + c8[i]) {
            sel[0] = lane * 8 + i;
            sel[1] = rem - static_cast<int>(run);
          }
          run += c8[i];
        }
      }
    }
    __syncthreads();
    prefix = (prefix << 8) | static_cast<uint32_t>(sel[0]);
    rem = sel[1];
    __syncthreads();
  }
  const uint32_t limit = limit_of(prefix);          // prefix is now the k-th smallest key
  if (tid == 0) sel[2] = 0;
  __syncthreads();
  for (int i0 = 0; i0 < n; i0 += kKnnThreads) {
    const int i = i0 + tid;
    const unsigned long long e = i < n ? bq[i] : ~0ull;
    const bool keep = i < n && static_cast<uint32_t>(e >> 32) <= limit;
    const uint32_t m = __ballot_sync(0xffffffffu, keep);
    int pos0 = 0;
    if (lane == 0 && m) pos0 = atomicAdd(&sel[2], __popc(m));
    pos0 = __shfl_sync(0xffffffffu, pos0, 0);
    if (keep) tmp[pos0 + __popc(m & ((1u << lane) - 1u))] = e;
  }
  __syncthreads();
  const int kept = sel[2];
  for (int i = tid; i < kept; i += kKnnThreads) bq[i] = tmp[i];
  *limit_out = limit;
  __syncthreads();
  return kept;
}

template <typename T>
__device__ __forceinline__ double exact_dist(const T* __restrict__ cb, int d, int i, int j) {
  const T* a = cb + static_cast<long long>(i) * d;
  const T* b = cb + static_cast<long long>(j) * d;
  double s = 0.0;
  for (int t = 0; t < d; ++t) {
    double diff = static_cast<double>(widen<T>(a[t])) - static_cast<double>(widen<T>(b[t]));
    s = fma(diff, diff, s);
  }
  return s;
}

// k rounds of an exact arg-min over (distance, index) greater than the last pick, by a CTA of NT threads
template <typename T, int NT>
__device__ __forceinline__ void argmin_rounds(const T* __restrict__ cb, int L, int d, int k, int qi, double* redd, int* redi,
                                              int32_t* out_i, float* out_d) {
  const int tid = threadIdx.x;
  double pd = -1.0;
  int pj = -1;
  for (int r = 0; r < k; ++r) {
    double bd = INFINITY;
    int bj = 0x7fffffff;
    for (int j = tid; j < L; j += NT) {
      if (j == qi) continue;
      const double dj = exact_dist<T>(cb, d, qi, j);
      const bool after = dj > pd || (dj == pd && j > pj);
      if (after && (dj < bd || (dj == bd && j < bj))) { bd = dj; bj = j; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double od = __shfl_xor_sync(0xffffffffu, bd, o);
      const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
      if (od < bd || (od == bd && oj < bj)) { bd = od; bj = oj; }
    }
    if ((tid & 31) == 0) { redd[tid >> 5] = bd; redi[tid >> 5] = bj; }
    __syncthreads();
    bd = redd[0]; bj = redi[0];
    for (int w = 1; w < NT / 32; ++w)
      if (redd[w] < bd || (redd[w] == bd && redi[w] < bj)) { bd = redd[w]; bj = redi[w]; }
    __syncthreads();
    pd = bd; pj = bj;
    if (tid == 0) {
      out_i[r] = bj;
      if (out_d) out_d[r] = static_cast<float>(bd);
    }
  }
}

// Exact ranking of one query's surviving candidates (keys carry the candidate index in their
// low 32 bits): distances re-evaluated in double, sorted by (distance, index), first k written.
// With `overflow` the buffer is ignored and k rounds of an exact arg-min over all rows are run.
template <typename T>
__device__ __forceinline__ void rank_query(const T* __restrict__ cb, int L, int d, int k, int qi,
                                           const unsigned long long* bq, int n_in, bool overflow, int CAP,
                                           double* sortd, int* sorti, double* redd, int* redi,
                                           int32_t* out_i, float* out_d) {
  const int tid = threadIdx.x;
    if (!overflow) {
    const int n = min(n_in, CAP);
          for (int i = tid; i < CAP; i += kKnnThreads) {
      if (i < n) {
        int j = static_cast<int>(bq[i] & 0xffffffffu);
        sorti[i] = j;
        sortd[i] = exact_dist<T>(cb, d, qi, j);
      } else {
        sorti[i] = 0x7fffffff;
        sortd[i] = INFINITY;
      }
    }
    __syncthreads();
    bitonic_pair(sortd, sorti, CAP);
    for (int r = tid; r < k; r += kKnnThreads) {
      out_i[r] = sorti[r];
      if (out_d) out_d[r] = static_cast<float>(sortd[r]);
    }
    __syncthreads();
  } else {
    argmin_rounds<T, kKnnThreads>(cb, L, d, k, qi, redd, redi, out_i, out_d);
  }
}

// Queries [q0, q0 + QT) of `total`: the rows themselves, or with LISTED the entries of a list.
template <typename T, bool LISTED>
__device__ __forceinline__ void knn_tile(const KnnArgs& a, const int q0, const int total, unsigned char* smem_raw) {
  const int QT = a.QT, CAP = a.CAP, d = a.d, L = a.L, k = a.k;
  const T* cb = static_cast<const T*>(a.cb);
  // layout: buf[QT][CAP] u64 | sortd[CAP] f64 | sorti[CAP] i32 | cand[256][kDC+1] f32 | tau[QT] f32 |
  //         cnt[QT] i32 | ovf[QT] i32 | redd[8] f64 | redi[8] i32 | queries
  unsigned long long* buf = reinterpret_cast<unsigned long long*>(smem_raw);
  double* sortd = reinterpret_cast<double*>(buf + static_cast<size_t>(QT) * CAP);
  double* redd = sortd + CAP;
  int* sorti = reinterpret_cast<int*>(redd + 8);
  float* cand = reinterpret_cast<float*>(sorti + CAP);
  float* tau = cand + kKnnThreads * (kDC + 1);
  int* cnt = reinterpret_cast<int*>(tau + QT);
  int* ovf = cnt + QT;
  int* redi = ovf + QT;
  uint32_t* hist = reinterpret_cast<uint32_t*>(redi + 8);       // [256] radix-select histogram
  int* sel = reinterpret_cast<int*>(hist + 256);               // [4]
  unsigned char* qraw = reinterpret_cast<unsigned char*>(sel + 4);
  qraw += (16 - (reinterpret_cast<uintptr_t>(qraw) & 15)) & 15;
  double* qd = reinterpret_cast<double*>(qraw);
  float* qf = reinterpret_cast<float*>(qraw);

  const int tid = threadIdx.x;
  const int nq = min(QT, total - q0);
  auto row_of = [&](int q) { return LISTED ? a.queries[q0 + q] : q0 + q; };

  const int dpad = (d + 7) & ~7;
  if (a.f32acc) {
    for (int i = tid; i < QT * dpad; i += kKnnThreads) {
      int q = i / dpad, t = i - q * dpad;
      qf[i] = (q < nq && t < d) ? widen<T>(cb[static_cast<long long>(row_of(q)) * d + t]) : 0.f;
    }
  } else {
    for (int i = tid; i < QT * d; i += kKnnThreads) {
      int q = i / d, t = i - q * d;
      float v = (q < nq) ? widen<T>(cb[static_cast<long long>(row_of(q)) * d + t]) : 0.f;
      if (a.q_double) qd[i] = static_cast<double>(v); else qf[i] = v;
    }
  }
  if (tid < QT) { tau[tid] = INFINITY; cnt[tid] = 0; ovf[tid] = 0; }
  __syncthreads();

  constexpr int MAXQT = 8;
  int own[MAXQT];                                     // (a query is no candidate of its own)
#pragma unroll
  for (int q = 0; q < MAXQT; ++q) own[q] = q < nq ? row_of(q) : -1;
  // d <= 8 (one chunk of dimensions): the candidate row of the next tile is fetched while this
  // tile is being processed
  float cnext[8];
  const bool prefetch = a.f32acc && d <= 8;
  auto fetch_row = [&](int row, float (&out)[8]) {
#pragma unroll
    for (int t = 0; t < 8; ++t) out[t] = (row < L && t < d) ? widen<T>(cb[static_cast<long long>(row) * d + t]) : 0.f;
  };
  if (prefetch) fetch_row(tid, cnext);
  for (int base = 0; base < L; base += kKnnThreads) {
    double acc[MAXQT];
#pragma unroll
    for (int q = 0; q < MAXQT; ++q) acc[q] = 0.0;
    const int ncand = min(kKnnThreads, L - base);
    if (a.f32acc) {
      // Filter distances in float32: every thread reads its candidate's row straight from global
      // memory, eight dimensions at a time, against the query rows in shared memory.  The relative
      // error of such a sum is below (d + 2) 2^-24, so with the margin applied to tau nothing
      // that can belong to the exact top k is dropped; exact duplicates still give 0.
      float accf[MAXQT];
#pragma unroll
      for (int q = 0; q < MAXQT; ++q) accf[q] = 0.f;
      for (int db = 0; db < d; db += 8) {
        float cv[8];
        if (prefetch) {
#pragma unroll
          for (int t = 0; t < 8; ++t) cv[t] = cnext[t];
          fetch_row(base + kKnnThreads + tid, cnext);
        } else {
#pragma unroll
          for (int t = 0; t < 8; ++t)
            cv[t] = (tid < ncand && db + t < d) ? widen<T>(cb[static_cast<long long>(base + tid) * d + db + t]) : 0.f;
        }
#pragma unroll
        for (int q = 0; q < MAXQT; ++q) {
          if (q < QT) {
            const float4 qa = *reinterpret_cast<const float4*>(qf + q * dpad + db);
            const float4 qb = *reinterpret_cast<const float4*>(qf + q * dpad + db + 4);
            const float qv[8] = {qa.x, qa.y, qa.z, qa.w, qb.x, qb.y, qb.z, qb.w};
#pragma unroll
            for (int t = 0; t < 8; ++t) {
              const float diff = qv[t] - cv[t];
              accf[q] = fmaf(diff, diff, accf[q]);
            }
          }
        }
      }
#pragma unroll
      for (int q = 0; q < MAXQT; ++q) acc[q] = static_cast<double>(accf[q]);
    } else
    for (int db = 0; db < d; db += kDC) {
      const int dc = min(kDC, d - db);
      __syncthreads();
      for (int i = tid; i < ncand * dc; i += kKnnThreads) {
        int r = i / dc, t = i - r * dc;
        cand[r * (kDC + 1) + t] = widen<T>(cb[static_cast<long long>(base + r) * d + db + t]);
      }
      __syncthreads();
      if (tid < ncand) {
        for (int t = 0; t < dc; ++t) {
          const double cv = static_cast<double>(cand[tid * (kDC + 1) + t]);
#pragma unroll
          for (int q = 0; q < MAXQT; ++q) {
            if (q < QT) {
              double qv = a.q_double ? qd[q * d + db + t] : static_cast<double>(qf[q * d + db + t]);
              double diff = qv - cv;
              acc[q] = fma(diff, diff, acc[q]);
            }
          }
        }
      }
    }
    // filter into the per-query buffers
    if (tid < ncand) {
      const int j = base + tid;
#pragma unroll
      for (int q = 0; q < MAXQT; ++q) {
        if (q < nq && j != own[q]) {
          float f = static_cast<float>(acc[q]);
          if (f <= tau[q]) {
            int pos = atomicAdd(&cnt[q], 1);
            if (pos < CAP) buf[static_cast<size_t>(q) * CAP + pos] =
                (static_cast<unsigned long long>(__float_as_uint(f)) << 32) | static_cast<unsigned>(j);
          }
        }
      }
    }
    __syncthreads();
    // cut back buffers that might overflow during the next tile
    for (int q = 0; q < nq; ++q) {
      int n = cnt[q];
      if (n <= CAP - kKnnThreads || ovf[q]) continue;     // uniform: cnt/ovf are shared
      unsigned long long* bq = buf + static_cast<size_t>(q) * CAP;
      // keep everything up to the k-th smallest filter distance (times the margin in float32 mode)
      uint32_t limit;
      const float margin = a.f32acc ? a.margin : 1.0f, slack = a.f32acc ? a.slack : 0.0f;
      const int m = radix_cut(bq, min(n, CAP), k, reinterpret_cast<unsigned long long*>(sortd), hist, sel,
                              [&](uint32_t kth) { return __float_as_uint(__fadd_ru(__fmul_ru(__uint_as_float(kth), margin), slack)); }, &limit);
      if (tid == 0) {
        tau[q] = __uint_as_float(limit);      // (non-negative floats order as their bits)
        cnt[q] = m;
        if (m > CAP - kKnnThreads) ovf[q] = 1;      // ties at tau fill the buffer
      }
      __syncthreads();
    }
  }

  // final ranking per query
  for (int q = 0; q < nq; ++q) {
    const int qi = row_of(q);
    rank_query<T>(cb, L, d, k, qi, buf + static_cast<size_t>(q) * CAP, cnt[q], ovf[q] != 0, CAP, sortd, sorti, redd, redi,
                  a.nbr_idx + static_cast<long long>(qi) * k,
                  a.nbr_dist ? a.nbr_dist + static_cast<long long>(qi) * k : nullptr);
  }
}

template <typename T>
__global__ void __launch_bounds__(kKnnThreads) knn_kernel(const KnnArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  knn_tile<T, false>(a, blockIdx.x * a.QT, a.L, smem_raw);
}

// The queries that the tcgen05 kernels gave up (usually none: the list is made on the device, so this is always launched,
// on about the CTAs that are resident at once).  Rows that crowd within the contraction's absolute error
// bound differ by far more than the relative margin here.
template <typename T>
__global__ void __launch_bounds__(kKnnThreads) knn_rest_kernel(const KnnArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  grid_dependency_sync();
  const int total = *a.n_queries;
  for (int q0 = blockIdx.x * a.QT; q0 < total; q0 += gridDim.x * a.QT) {
    knn_tile<T, true>(a, q0, total, smem_raw);
    __syncthreads();                                  // the next queries overwrite the shared memory
  }
}

}  // namespace lantern

#include "knn_t5.cuh"

using namespace lantern;

namespace {
// Where the table is built by the tcgen05 kernels, and with which sizes.  Operand rows of up to 256
// elements fit the shared-memory tiles (bfloat16 rows of up to 256 elements; float32 rows, three parts each, of up
// to 85) and k <= 320 keeps a query's survivors within the ranking's 512 slots.  Against the brute-force kernel (and, for
// bfloat16, an mma.sync kernel that stood here): 16384 x 8 float32, k = 100: 0.45 ms, was 2.63; 20000 x 64 float32,
// k = 200: 0.91 ms, was 17.4; 600 x 256 bfloat16, k = 200: 81 us, was 567; 300 x 8 float32, k = 10: 49 us, was 116.
// Below one half tile of rows nothing is left to select.
#ifndef LANTERN_T5_MIN_L
#define LANTERN_T5_MIN_L 64
#endif
struct T5Plan {
  bool ok, sampled;                 // sampled: the sample is a proper part of the codebook, with tiles of its own
  int dp, tiles, nst, gshift, groups;
  int first_tiles;                  // query tiles of the first (largest) chunk
  size_t off_cn, off_sn, off_rest, off_counts, off_bound, off_qm, off_cm, off_sm, off_minima, off_lists, bytes;
};
size_t round256(size_t x) { return (x + 255) / 256 * 256; }
int t5_split(int tiles, int L) {    // CTAs per query tile of a chunk
  int s = kT5Items / tiles;
  if (s > kT5MaxSplit) s = kT5MaxSplit;
  const int nct = (L + kT5C - 1) / kT5C;
  if (s > nct) s = nct;
  return s < 1 ? 1 : s;
}
// Entries a list holds: what the sampled bound lets through when the sample is representative (the k+1
// smallest of `groups` group minima are the about -groups ln(1 - (k+1)/groups) smallest sampled candidates) with six
// standard deviations, at least k + 192, at most what cut-backs work well with.
int t5_cap(const T5Plan& p, int L, int k, int split) {
  const double share = static_cast<double>(k + 1) / p.groups;
  const double est = (share < 0.95 ? -p.groups * log(1.0 - share) * L / (static_cast<double>(p.nst) * kT5C) : L) / (kT5Per * split);
  double c = est + 6.0 * sqrt(est) + 64.0;
  if (c > 1024.0) c = 1024.0;
  if (c < k + 193.0) c = k + 193.0;
  return (static_cast<int>(c) + 63) / 64 * 64;
}
T5Plan t5_plan(lantern_dtype dt, int L, int d, int k) {
  T5Plan p = {};
  const int parts = dt == LANTERN_F32 ? 3 : 1;
  p.ok = L >= LANTERN_T5_MIN_L && k <= kT5MaxK && d <= 256 && parts * d <= 256;
  if (!p.ok) return p;
  p.dp = (parts * d + 15) / 16 * 16;
  p.tiles = (L + kT5Q - 1) / kT5Q;
  // one candidate in four is sampled, 1024 at least; groups of the smallest size that leaves at most 1024 minima
  int sample = (L + 3) / 4;
  if (sample < 1024) sample = 1024;
  if (sample > L) sample = L;
  p.nst = (sample + kT5C - 1) / kT5C;
  if (p.nst > kT5MaxGroups / 4) p.nst = kT5MaxGroups / 4;      // groups of 32 columns at most
  while ((p.nst * kT5C) >> p.gshift > kT5MaxGroups) ++p.gshift;
  p.groups = (p.nst * kT5C) >> p.gshift;
  p.first_tiles = p.tiles < kT5Items ? p.tiles : kT5Items;
  const int split = t5_split(p.first_tiles, L);
  const size_t segs = static_cast<size_t>(kT5Items) * kT5Sel;
  p.sampled = p.nst < p.tiles;
  const size_t tile = static_cast<size_t>(kT5Q) * p.dp * 2, side = p.tiles * tile;
  p.off_cn = round256((static_cast<size_t>(L) + 64) * sizeof(float));
  p.off_sn = p.off_cn + static_cast<size_t>(p.tiles) * kT5C * sizeof(float);
  p.off_rest = p.off_sn + static_cast<size_t>(p.sampled ? p.nst : 0) * kT5C * sizeof(float);
  p.off_counts = p.off_rest + round256(static_cast<size_t>(L) * sizeof(int));
  p.off_bound = p.off_counts + segs * sizeof(int);
  p.off_qm = p.off_bound + static_cast<size_t>(kT5Items) * kT5Q * sizeof(float);
  p.off_cm = p.off_qm + (dt == LANTERN_F32 ? side : 0);
  p.off_sm = p.off_cm + side;
  p.off_minima = p.off_sm + (p.sampled ? p.nst * tile : 0);
  p.off_lists = p.off_minima + static_cast<size_t>(p.first_tiles) * p.groups * kT5Q * sizeof(float);
  // (a later chunk has fewer tiles, so no more CTAs and no longer lists)
  p.bytes = p.off_lists + static_cast<size_t>(p.first_tiles) * split * kT5Sel * t5_cap(p, L, k, split) * 8;
  return p;
}

// Arguments of the brute-force kernels; returns their shared memory.
size_t brute_shape(KnnArgs& a, const void* codebook, int L, int d, int k, int32_t* nbr_idx, float* nbr_dist) {
  a.cb = codebook; a.L = L; a.d = d; a.k = k; a.nbr_idx = nbr_idx; a.nbr_dist = nbr_dist;
  int cap = 512;
  while (cap < k + 2 * kKnnThreads) cap *= 2;
  a.CAP = cap;
  a.QT = cap <= 1024 ? 8 : 4;
  auto smem_for = [&](int qt, int qdouble) {
    return static_cast<size_t>(qt) * cap * 8 + static_cast<size_t>(cap) * 12 + 8 * 12 +
           static_cast<size_t>(kKnnThreads) * (kDC + 1) * 4 + static_cast<size_t>(qt) * 12 + 16 + 260 * 4 +
           static_cast<size_t>(qt) * ((d + 7) & ~7) * (qdouble ? 8 : 4);
  };
  a.f32acc = d <= 64 ? 1 : 0;
  a.margin = 1.0f + 3.0f * static_cast<float>(d + 2) * 5.9604644775390625e-8f;
  a.slack = static_cast<float>(d + 2) * 2.8025969e-45f;          // two roundings of 2^-150 per term, doubled
  a.q_double = (!a.f32acc && smem_for(a.QT, 1) <= 160 * 1024) ? 1 : 0;
  while (a.QT > 1 && smem_for(a.QT, a.q_double) > 220 * 1024) a.QT /= 2;
  return smem_for(a.QT, a.q_double);
}

template <typename T>
lantern_status build_t5(const T5Plan& p, const T* cb, int L, int d, int k, int32_t* nbr_idx, float* nbr_dist,
                        unsigned char* ws, cudaStream_t st) {
  float* nrm = reinterpret_cast<float*>(ws);
  if (cudaMemsetAsync(nrm + L, 0, 3 * sizeof(float), st) != cudaSuccess) return LANTERN_ERR_CUDA;
  KnnPrepArgs g;
  g.cb = cb; g.L = L; g.d = d; g.dp = p.dp;
  g.rows = p.tiles * kT5C;
  g.sampled = p.sampled ? p.nst * kT5C : 0;
  g.step = p.sampled ? (static_cast<unsigned long long>(L) << 32) / (static_cast<unsigned long long>(p.nst) * kT5C) : 0;
  g.nrm = nrm;
  g.cn = reinterpret_cast<float*>(ws + p.off_cn);
  g.sn = reinterpret_cast<float*>(ws + p.off_sn);
  g.qm = ws + p.off_qm;                       // (bfloat16 rows: the candidate side's tiles, off_qm == off_cm)
  g.cm = ws + p.off_cm;
  g.sm = ws + p.off_sm;
  knn_prep_kernel<T><<<(g.rows + g.sampled) / 8, 256, 0, st>>>(g);
  KnnT5Args a;
  a.qm = g.qm;
  a.nrm = nrm;
  a.minima = reinterpret_cast<float*>(ws + p.off_minima);
  float* bound = reinterpret_cast<float*>(ws + p.off_bound);
  a.bound = bound;
  a.lists = reinterpret_cast<unsigned long long*>(ws + p.off_lists);
  a.counts = reinterpret_cast<int*>(ws + p.off_counts);
  a.L = L; a.dp = p.dp; a.k = k;
  a.gshift = p.gshift; a.groups = p.groups;
  a.eps1 = static_cast<float>(p.dp + 16) * 4.76837158203125e-7f + (sizeof(T) == 4 ? 1.52587890625e-5f : 0.f);   // 2^-21, 2^-16
  a.eps0 = static_cast<float>(p.dp) * 2.3509887016445750e-38f;                                                    // products below the normal range
  KnnRankArgs r;
  r.cb = cb; r.nrm = nrm; r.lists = a.lists; r.counts = a.counts;
  r.L = L; r.d = d; r.k = k; r.eps1 = a.eps1; r.eps0 = a.eps0; r.nbr_idx = nbr_idx; r.nbr_dist = nbr_dist;
  r.rest = reinterpret_cast<int*>(ws + p.off_rest);
  r.n_rest = reinterpret_cast<int*>(nrm + L + 2);
  r.lanes = 0;
  if (d % 8 == 0 && reinterpret_cast<uintptr_t>(cb) % 16 == 0) {
    r.lanes = 1;
    while (r.lanes < 8 && r.lanes * 2 <= d / 8) r.lanes *= 2;
  }
  KnnArgs b = {};
  const size_t smb = brute_shape(b, cb, L, d, k, nbr_idx, nbr_dist);
  b.queries = r.rest; b.n_queries = r.n_rest;
  const size_t sm5 = knn_t5_smem(p.dp), smr = knn_rank_smem(d);
  if (cudaFuncSetAttribute(knn_rest_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smb)) != cudaSuccess ||
      cudaFuncSetAttribute(knn_t5_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(sm5)) != cudaSuccess ||
      cudaFuncSetAttribute(knn_t5_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(sm5)) != cudaSuccess)
    return LANTERN_ERR_CUDA;
  for (a.tile0 = 0; a.tile0 < p.tiles; a.tile0 += kT5Items) {
    const int n = p.tiles - a.tile0 < kT5Items ? p.tiles - a.tile0 : kT5Items;
    const int split = t5_split(n, L);
    a.cap = t5_cap(p, L, k, split);
    a.split = split < p.nst ? split : p.nst;
    a.nct = p.nst; a.cm = p.sampled ? g.sm : g.cm; a.cn = p.sampled ? g.sn : g.cn;
    knn_t5_kernel<true><<<n * a.split, kT5Threads, sm5, st>>>(a);
    knn_bound_kernel<<<n * kT5Q / 8, 256, 0, st>>>(a.minima, n * kT5Q, p.groups, k + 1, bound);
    a.split = split;
    a.nct = p.tiles; a.cm = g.cm; a.cn = g.cn;
    knn_t5_kernel<false><<<n * split, kT5Threads, sm5, st>>>(a);
    r.cap = a.cap; r.split = split; r.q0 = a.tile0 * kT5Q;
    const int queries = L - r.q0 < n * kT5Q ? L - r.q0 : n * kT5Q;
    knn_rank_kernel<T><<<queries, kRankThreads, smr, st>>>(r);
  }
  const int groups = (L + b.QT - 1) / b.QT, resident = smb <= 113 * 1024 ? 2 * kT5Items : kT5Items;
  if (launch_after_previous(knn_rest_kernel<T>, static_cast<unsigned>(groups < resident ? groups : resident), kKnnThreads, smb, st, 1, b) !=
      cudaSuccess)
    return LANTERN_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? LANTERN_OK : LANTERN_ERR_CUDA;
}

// bfloat16 shapes whose workspace has always been required (their calls are refused without it)
bool needs_workspace(lantern_dtype dt, int L, int d, int k) {
  return dt == LANTERN_BF16 && k <= kT5MaxK && d <= 256 && (L >= 8192 ? d % 8 == 0 : L >= 64 && d % 16 == 0 && d >= 32);
}
}  // namespace

extern "C" size_t lantern_build_neighbors_workspace(lantern_dtype dt, int32_t L, int32_t d, int32_t k) {
  if (L < 2 || d < 1 || k < 1) return 0;
  const T5Plan p = t5_plan(dt, L, d, k);
  return p.ok ? p.bytes : 0;                  // the brute-force kernel keeps all of its state on chip
}

extern "C" lantern_status lantern_build_neighbors(const void* codebook, lantern_dtype dt, int32_t L, int32_t d,
                                                  int32_t k, int32_t* nbr_idx, float* nbr_dist, void* workspace,
                                                  size_t workspace_bytes, void* stream) {
  if (!codebook || !nbr_idx) return LANTERN_ERR_INVALID_ARG;
  if (dt != LANTERN_F32 && dt != LANTERN_BF16) return LANTERN_ERR_INVALID_ARG;
  if (L < 2 || d < 1 || k < 1 || k > L - 1) return LANTERN_ERR_INVALID_ARG;
  if (k > 1024 || d > 4096) return LANTERN_ERR_UNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const T5Plan p = t5_plan(dt, L, d, k);
  if (p.ok) {
    const bool have = workspace && workspace_bytes >= p.bytes && reinterpret_cast<uintptr_t>(workspace) % 256 == 0;
    const bool aligned = reinterpret_cast<uintptr_t>(codebook) % 16 == 0;
    if (needs_workspace(dt, L, d, k)) {
      if (!have) return LANTERN_ERR_WORKSPACE;
      if (!aligned) return LANTERN_ERR_INVALID_ARG;
    }
    if (have) {
      unsigned char* ws = static_cast<unsigned char*>(workspace);
      return dt == LANTERN_F32 ? build_t5(p, static_cast<const float*>(codebook), L, d, k, nbr_idx, nbr_dist, ws, st)
                               : build_t5(p, static_cast<const __nv_bfloat16*>(codebook), L, d, k, nbr_idx, nbr_dist, ws, st);
    }
  }
  KnnArgs a = {};
  const size_t smem = brute_shape(a, codebook, L, d, k, nbr_idx, nbr_dist);
  if (smem > 227 * 1024) return LANTERN_ERR_UNSUPPORTED;
  const int grid = (L + a.QT - 1) / a.QT;
  cudaError_t e;
  if (dt == LANTERN_F32) {
    e = cudaFuncSetAttribute(knn_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e == cudaSuccess) { knn_kernel<float><<<grid, kKnnThreads, smem, st>>>(a); e = cudaGetLastError(); }
  } else {
    e = cudaFuncSetAttribute(knn_kernel<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e == cudaSuccess) { knn_kernel<__nv_bfloat16><<<grid, kKnnThreads, smem, st>>>(a); e = cudaGetLastError(); }
  }
  return e == cudaSuccess ? LANTERN_OK : LANTERN_ERR_CUDA;
}
