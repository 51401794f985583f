// Dynamic-tree drafting (Sec. 2.1, the dynamic variant of tree drafting; Sec. 3 "Shallow draft trees"):
// every draft node carries log V = sum of the logs of the drafter's confidences along its path.
//   expand_rows_kernel   one CTA per frontier node: the K most confident tokens of its drafter row
//                        become candidates (token, parent, log V, depth) in the sequence's pool;
//   select_frontier_kernel  one CTA per sequence: the E candidates of this depth with the largest
//                        log V form the next frontier;
//   trim_tree_kernel     one CTA per sequence: the m - 1 pool entries with the largest log V and
//                        the root, renumbered breadth first (the numbering lantern_tree_create wants).
// Orders of equal values: tokens of a row by (z descending, token ascending), candidates by
// (log V descending, pool index ascending); a parent therefore always ranks before its children.
#include <cmath>

#include "toplist.cuh"

namespace lantern {

constexpr int kDynThreads = 256;
constexpr int kDynMaxPool = 2048;

struct ExpandArgs {
  const void *dc, *du;
  long long row_stride, seq_stride;
  int B, F, K, E, V, allow_lo, allow_hi;
  float g, inv_tau;
  const int32_t* frontier;           // [B][F] pool index of the node in each slot, -1: empty slot
  int P, pool_off, depth;
  int32_t *pool_parent, *pool_token, *pool_depth;
  double* pool_logv;
  int32_t* next_frontier;            // [B][E]
};

// (value, index) maximum with ties to the lower index, over the CTA; result in every thread
__device__ __forceinline__ void block_best(float& z, int& j, float* sz, int* sj) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float oz = __shfl_xor_sync(0xffffffffu, z, o);
    const int oj = __shfl_xor_sync(0xffffffffu, j, o);
    if (oz > z || (oz == z && oj < j)) { z = oz; j = oj; }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) { sz[warp] = z; sj[warp] = j; }
  __syncthreads();
  z = sz[0]; j = sj[0];
  for (int w = 1; w < kDynThreads / 32; ++w)
    if (sz[w] > z || (sz[w] == z && sj[w] < j)) { z = sz[w]; j = sj[w]; }
  __syncthreads();
}

// The round of the fallback path: best token after (pz, pj) over the whole row, scalar loads.  Kept out
// of line so that this rarely used scan does not grow the kernel's main loops.
template <typename T>
__device__ __noinline__ void scan_row_after(const T* c, const T* u, float g, float inv_tau, int lo, int hi, float pz, int pj,
                                            float& bz, int& bj) {
  for (int j = lo + threadIdx.x; j < hi; j += kDynThreads) {
    const float z = u ? combine<true>(Vec<T>::widen(c[j]), Vec<T>::widen(u[j]), g, inv_tau)
                      : combine<false>(Vec<T>::widen(c[j]), 0.f, g, inv_tau);
    const bool after = z < pz || (z == pz && j > pj);
    if (after && (z > bz || (z == bz && j < bj))) { bz = z; bj = j; }
  }
}

// Softmax denominator of a thread's elements relative to a reference m (-inf: none yet): terms in float32 from exact
// differences, a vector's terms summed in float32 and folded into a double.  A term's argument is rounded to |z - m| 2^-24,
// which for z far above m is lost accuracy of a term that makes up the sum: an element more than kRefSlack above the
// reference becomes the reference, so that its own term is 1.
constexpr float kRefSlack = 1.f;
template <int VN>
__device__ __forceinline__ float sum_terms(const float (&z)[VN], float m) {
  float part = 0.f;
#pragma unroll
  for (int e = 0; e < VN; ++e) part += ex2_approx(__fmul_rn(__fsub_rn(z[e], m), kLog2e));
  return part;
}
template <int VN>
__device__ __forceinline__ void fold_exp(const float (&z)[VN], float& m, double& s) {
  float top = z[0];
#pragma unroll
  for (int e = 1; e < VN; ++e) top = fmaxf(top, z[e]);
  if (top > m + kRefSlack) {
    if (m > -INFINITY) s *= exp(static_cast<double>(m) - static_cast<double>(top));
    m = top;
  }
  s += static_cast<double>(sum_terms<VN>(z, m > -INFINITY ? m : 0.f));    // (no finite element so far: 0, or NaN for a NaN)
}

// One frontier row by one CTA, or by a cluster when a call has few rows: the row is streamed once.  The first
// chunk's elements give a threshold, a lower bound of the row's K-th largest value; the few elements that reach it go to
// a list in shared memory, cut back to its K best after a third of the row, and the softmax denominator comes from
// the same pass.  The CTAs of a row push their K best and their sums to the first one, which writes the
// children in the order (z descending, token ascending).
// Bound: instruction issue and the latency of a chunk's loads.  A depth (rows and frontier) of 512 rows of 65536 bfloat16
// logits: 33 us, with two passes over the row (maxima, then terms and list) 40; of 8 rows: 14 us, was 25; 512 rows of
// 40003 logits (most of them unaligned): 27 us, was 92.  (Six depths of 64 sequences and the trimming: 203 us; 199 with
// the terms relative to a thread's first maximum, which cost accuracy.)
template <typename T, bool CFG, bool TAU1>
__global__ void __launch_bounds__(kDynThreads, 4) expand_rows_kernel(const ExpandArgs a) {
  using namespace stream;
  static_assert(kDynThreads == ST, "the list helpers are built for this many threads");
  using IO = RowIO<T, CFG, TAU1>;
  constexpr int VN = IO::VN;
  constexpr int UV = (CFG ? 2 : 4) * 4 / VN;
  static_assert(ST * UV * VN <= kIterElems, "iteration size");
  grid_dependency_sync();
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  TopList s;
  s.list = reinterpret_cast<uint2*>(dyn_smem);
  s.fin = s.list + kListCap;
  s.pk = s.fin + kFinal;
  s.top = s.pk + 2 * 2 * SW;
  s.rinfo = s.top + 16;
  double* rsum = reinterpret_cast<double*>(s.rinfo + kMaxCluster);    // [kMaxCluster] the CTAs' sums, in CTA 0
  double* wsum = rsum + kMaxCluster;                                   // [SW] the warps' sums
  float* rmax = reinterpret_cast<float*>(wsum + SW);                   // [SW] the warps' references
  int* sj = reinterpret_cast<int*>(rmax + SW);                         // [SW]
  s.cnt = sj + SW;
  s.fkey = nullptr;
  const uint32_t rank = cluster_ctarank(), nrank = cluster_nctarank();
  if (nrank > 1) cluster_arrive_relaxed();            // waited for before the first access to a peer's shared memory
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int idx = blockIdx.x / nrank;
  const int b = idx / a.F, f = idx - b * a.F;
  const int node = a.frontier[b * a.F + f];
  const long long pbase = static_cast<long long>(b) * a.P + a.pool_off + f * a.K;
  if (node < 0) {                                   // empty slot: candidates that can never be chosen (the whole cluster leaves)
    if (rank == 0) {
      for (int r = tid; r < a.K; r += kDynThreads) {
        a.pool_parent[pbase + r] = -1;
        a.pool_token[pbase + r] = -1;
        a.pool_depth[pbase + r] = a.depth;
        a.pool_logv[pbase + r] = -INFINITY;
      }
    }
    if (nrank > 1) cluster_wait();
    return;
  }
  const int K = a.K;
  IO io;
  io.c = static_cast<const T*>(a.dc) + b * a.seq_stride + f * a.row_stride;
  io.u = CFG ? static_cast<const T*>(a.du) + b * a.seq_stride + f * a.row_stride : nullptr;
  io.g = a.g; io.it = a.inv_tau;
  // vectors from the 16-byte boundary at or before the first allowed token (rows need no alignment here); rows whose two
  // operands sit differently are read element by element
  Geo ge;
  ge.alo = a.allow_lo; ge.ahi = a.allow_hi;
  const int off = static_cast<int>((reinterpret_cast<uintptr_t>(io.c + ge.alo) & 15u) / sizeof(T));
  const bool together = !CFG || ((reinterpret_cast<uintptr_t>(io.c) ^ reinterpret_cast<uintptr_t>(io.u)) & 15u) == 0;
  ge.j0 = ge.alo - off;
  io.j0 = ge.j0;
  ge.nvec = (ge.ahi - ge.j0 + VN - 1) / VN;
  ge.vi0 = off > 0 ? 1 : 0;
  ge.vi1 = (ge.j0 + ge.nvec * VN > ge.ahi) ? ge.nvec - 1 : ge.nvec;
  if (ge.vi1 < ge.vi0 || !together) ge.vi1 = ge.vi0;
  const int nwarps = static_cast<int>(nrank) * SW;
  ge.vw = ((ge.nvec + nwarps - 1) / nwarps + 31) / 32 * 32;
  const int gw = static_cast<int>(rank) * SW + warp;
  const int vbeg = min(gw * ge.vw, ge.nvec), vend = min(vbeg + ge.vw, ge.nvec);
  if (tid == 0) *s.cnt = 0;
  __syncthreads();

  auto append = [&](float z, int tok) {
    const int pos = atomicAdd(s.cnt, 1);
    if (pos < kListCap) s.list[pos] = make_uint2(__float_as_uint(z), static_cast<uint32_t>(tok));
  };
  auto cut = [&](float T0) { return *s.cnt <= ST ? cut_ranked(s, K, T0) : cut_list(s, K, T0); };
  // z of vector vv (anything beyond the warp's range or the allowed tokens: -inf)
  auto vec_z = [&](int vv, const uint4& rc, const uint4& ru, float (&z)[VN]) {
    if (vv < vend && vv >= ge.vi0 && vv < ge.vi1) {
      io.z(rc, ru, z);
    } else {
#pragma unroll
      for (int e = 0; e < VN; ++e) {
        const int t = ge.j0 + vv * VN + e;
        z[e] = (vv < vend && t >= ge.alo && t < ge.ahi) ? io.z_at(t) : -INFINITY;
      }
    }
  };
  float Tk, m;
  double sum;
  const int iters = (ge.vw + 32 * UV - 1) / (32 * UV);
  const int cut_it = max(1, iters / 3);
  for (int mode = 0; mode < 2; ++mode) {              // (mode 1: the list overflowed, the row is redone with a cut after every chunk)
    m = -INFINITY;
    sum = 0.0;
    {
      uint4 rc[UV], ru[UV];
#pragma unroll
      for (int u = 0; u < UV; ++u) {
        const int vv = vbeg + 32 * u + lane;
        if (vv < vend && vv >= ge.vi0 && vv < ge.vi1) io.load(vv, rc[u], ru[u]);
      }
      float first[UV][VN];
      float tbk = -INFINITY;
      int tbj = 0x7fffffff;
#pragma unroll
      for (int u = 0; u < UV; ++u) {
        const int vv = vbeg + 32 * u + lane;
        vec_z(vv, rc[u], ru[u], first[u]);
#pragma unroll
        for (int e = 0; e < VN; ++e)
          if (key_before(first[u][e], ge.j0 + vv * VN + e, tbk, tbj)) { tbk = first[u][e]; tbj = ge.j0 + vv * VN + e; }
      }
      Tk = first_threshold(s, K, tbk, tbj);
      m = first_best(s);                               // the chunk's maximum: few elements of the row lie above it
#pragma unroll
      for (int u = 0; u < UV; ++u) {
        sum += static_cast<double>(sum_terms<VN>(first[u], m > -INFINITY ? m : 0.f));
#pragma unroll
        for (int e = 0; e < VN; ++e)
          if (first[u][e] >= Tk && first[u][e] > -INFINITY) append(first[u][e], ge.j0 + (vbeg + 32 * u + lane) * VN + e);
      }
    }
    if (mode == 1) {
      __syncthreads();
      const bool full = *s.cnt > kListCap - kIterElems;
      __syncthreads();
      if (full) Tk = cut(Tk);
    }
    for (int it = 1; it < iters; ++it) {
      const int base = vbeg + it * 32 * UV;
      constexpr int UF = 2 * UV;                       // two chunks at once where nothing has to be checked between them
      if (mode == 0 && it != cut_it && it + 1 < iters && base >= ge.vi0 && base + 32 * UF <= min(vend, ge.vi1)) {
        uint4 rc[UF], ru[UF];                          // whole vectors only, the same in every lane
#pragma unroll
        for (int u = 0; u < UF; ++u) io.load(base + 32 * u + lane, rc[u], ru[u]);
        uint32_t hit = 0u;                             // vectors with an entry for the list
        float part[UF], above = -INFINITY;
#pragma unroll
        for (int u = 0; u < UF; ++u) {
          float z[VN];
          io.z(rc[u], ru[u], z);
          float top = z[0];
#pragma unroll
          for (int e = 1; e < VN; ++e) top = fmaxf(top, z[e]);
          if (top >= Tk) hit |= 1u << u;
          above = fmaxf(above, top);
          part[u] = sum_terms<VN>(z, m);
        }
        if (above <= m + kRefSlack && m > -INFINITY) {  // (one check for all vectors: the reference stays)
#pragma unroll
          for (int u = 0; u < UF; ++u) sum += static_cast<double>(part[u]);
        } else {
#pragma unroll
          for (int u = 0; u < UF; ++u) {
            float z[VN];
            io.z(rc[u], ru[u], z);
            fold_exp<VN>(z, m, sum);
          }
        }
        while (hit) {                                  // few: the vector is read again, so that it need not be kept
          const int vv = base + 32 * (__ffs(hit) - 1) + lane;
          hit &= hit - 1u;
          uint4 c1, u1;
          io.load(vv, c1, u1);
          float z[VN];
          io.z(c1, u1, z);
#pragma unroll
          for (int e = 0; e < VN; ++e)
            if (z[e] >= Tk && z[e] > -INFINITY) append(z[e], ge.j0 + vv * VN + e);
        }
        ++it;
        if (it != cut_it) continue;
      } else {
#pragma unroll 1
        for (int u = 0; u < UV; ++u) {
          const int vv = base + 32 * u + lane;
          uint4 rc, ru;
          if (vv < vend && vv >= ge.vi0 && vv < ge.vi1) io.load(vv, rc, ru);
          float z[VN];
          vec_z(vv, rc, ru, z);
#pragma unroll
          for (int e = 0; e < VN; ++e)
            if (z[e] >= Tk && z[e] > -INFINITY) append(z[e], ge.j0 + vv * VN + e);
          fold_exp<VN>(z, m, sum);
        }
      }
      if (it == cut_it || mode == 1) {
        __syncthreads();
        const int cn = *s.cnt;
        __syncthreads();                                // everyone has read the count before it moves again
        if (cn <= kListCap && (mode == 1 ? cn > kListCap - kIterElems : cn > K)) Tk = cut(Tk);
      }
    }
    __syncthreads();
    const bool overflow = *s.cnt > kListCap;
    if (!overflow) break;
    __syncthreads();                                    // (mode 1 never overflows: it cuts in time)
    if (tid == 0) *s.cnt = 0;
    __syncthreads();
  }
  cut(Tk);
  // ---- the sums relative to the CTA's largest reference, in double precision
  {
    const float wm = warp_max(m);
    double v = m == wm || m == -INFINITY ? sum : sum * exp(static_cast<double>(m) - static_cast<double>(wm));   // (-inf: 0 or NaN)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) { wsum[warp] = v; rmax[warp] = wm; }
  }
  __syncthreads();
  float cm = -INFINITY;
  for (int w = 0; w < SW; ++w) cm = fmaxf(cm, rmax[w]);
  double cs = 0.0;
  if (tid == 0)
    for (int w = 0; w < SW; ++w)
      cs += rmax[w] != -INFINITY ? wsum[w] * exp(static_cast<double>(rmax[w]) - static_cast<double>(cm)) : wsum[w];
  int nf = *s.cnt;
  if (nrank > 1) {
    cluster_wait();                                   // every CTA of the row has started
    if (tid < nf) dsmem_st_u64(dsmem_addr(smem_u32(&s.fin[rank * kMaxR + tid]), 0), s.list[tid]);
    if (tid == 0) {
      dsmem_st_u64(dsmem_addr(smem_u32(&s.rinfo[rank]), 0), make_uint2(static_cast<uint32_t>(nf), __float_as_uint(cm)));
      const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(cs));
      dsmem_st_u64(dsmem_addr(smem_u32(&rsum[rank]), 0), make_uint2(static_cast<uint32_t>(bits), static_cast<uint32_t>(bits >> 32)));
    }
    cluster_sync();
    if (rank != 0) return;
    nf = merge_lists(s, nrank);
  }
  // ---- children: the first K of the order
  if (tid == 0) {
    const float top = nf > 0 ? __uint_as_float(s.list[0].x) : -INFINITY;          // the row's maximum
    double total = 0.0;
    if (nrank > 1) {
      for (uint32_t r = 0; r < nrank; ++r) {
        const float rm = __uint_as_float(s.rinfo[r].y);
        total += rm != -INFINITY ? rsum[r] * exp(static_cast<double>(rm) - static_cast<double>(top)) : rsum[r];
      }
    } else {
      total = cm != -INFINITY ? cs * exp(static_cast<double>(cm) - static_cast<double>(top)) : cs;
    }
    // at least the top's own term, 1: its float32 stand-in may have lost a few units, and a child's log V never
    // rises above its parent's (which trimming relies on).  (A NaN stays one.)
    wsum[0] = total < 1.0 ? 0.0 : log(total);
    wsum[1] = a.pool_logv[static_cast<long long>(b) * a.P + node];
  }
  __syncthreads();
  const float bm = nf > 0 ? __uint_as_float(s.list[0].x) : -INFINITY;
  const double ln_s = wsum[0], parent_logv = wsum[1];
  auto child = [&](int r, float z, int tok, bool found) {      // fewer than K allowed tokens: the rest can never be chosen
    a.pool_parent[pbase + r] = found ? node : -1;
    a.pool_token[pbase + r] = found ? tok : -1;
    a.pool_depth[pbase + r] = a.depth;
    a.pool_logv[pbase + r] = found ? parent_logv + ((static_cast<double>(z) - static_cast<double>(bm)) - ln_s) : -INFINITY;
  };
  if (tid < min(nf, K)) child(tid, __uint_as_float(s.list[tid].x), static_cast<int>(s.list[tid].y), true);
  if (nf < K) {                                       // (fewer finite logits than children: tokens without mass, by token)
    float pz = nf > 0 ? __uint_as_float(s.list[nf - 1].x) : INFINITY;
    int pj = nf > 0 ? static_cast<int>(s.list[nf - 1].y) : -1;
    for (int r = nf; r < K; ++r) {
      float bz = -INFINITY;
      int bj = 0x7fffffff;
      scan_row_after<T>(io.c, io.u, a.g, a.inv_tau, a.allow_lo, a.allow_hi, pz, pj, bz, bj);
      block_best(bz, bj, rmax, sj);
      if (tid == 0) child(r, bz, bj, bj != 0x7fffffff);
      pz = bz;
      pj = bj;
    }
  }
}
__host__ __device__ constexpr size_t expand_smem() {
  return (stream::kListCap + stream::kFinal + 2 * 2 * stream::SW + 16 + kMaxCluster) * 8 + (kMaxCluster + stream::SW) * 8 +
         stream::SW * 8 + 16;
}

// order-preserving map of a double to an unsigned 64-bit integer (compares then run on the integer pipe)
__device__ __forceinline__ unsigned long long mono64(double x) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// rank of entry i among n entries by (value descending, index ascending); v holds mono64 keys
__device__ __forceinline__ int rank_desc(const unsigned long long* v, int n, int i) {
  const unsigned long long vi = v[i];
  int r = 0;
#pragma unroll 8
  for (int j = 0; j < n; ++j) {
    const unsigned long long vj = v[j];
    r += (vj > vi || (vj == vi && j < i)) ? 1 : 0;
  }
  return r;
}

__global__ void __launch_bounds__(kDynThreads) select_frontier_kernel(const ExpandArgs a) {
  grid_dependency_sync();
  extern __shared__ unsigned long long dyn_lv[];
  const int b = blockIdx.x, tid = threadIdx.x, T = a.F * a.K;
  const double* lv = a.pool_logv + static_cast<long long>(b) * a.P + a.pool_off;
  for (int i = tid; i < T; i += kDynThreads) dyn_lv[i] = mono64(lv[i]);
  for (int e = tid; e < a.E; e += kDynThreads) a.next_frontier[b * a.E + e] = -1;
  __syncthreads();
  for (int i = tid; i < T; i += kDynThreads) {
    if (dyn_lv[i] == mono64(-INFINITY)) continue;
    const int r = rank_desc(dyn_lv, T, i);
    if (r < a.E) a.next_frontier[b * a.E + r] = a.pool_off + i;
  }
}

struct TrimArgs {
  int B, P, used, m, max_depth;
  const int32_t *pool_parent, *pool_token, *pool_depth;
  const double* pool_logv;
  int32_t *n_nodes, *parent, *token, *pool_index;
  double* logv;
};

__global__ void __launch_bounds__(kDynThreads) trim_tree_kernel(const TrimArgs a) {
  grid_dependency_sync();
  extern __shared__ unsigned long long dyn_lv[];     // [used] keys of log V | new id | selected | depth | parent, [used] each
  int* newid = reinterpret_cast<int*>(dyn_lv + a.used);
  int* sel = newid + a.used;
  int* dep_s = sel + a.used;
  int* par_s = dep_s + a.used;
  __shared__ int count, level_n;
  const int b = blockIdx.x, tid = threadIdx.x, n = a.used;
  const long long base = static_cast<long long>(b) * a.P;
  for (int i = tid; i < n; i += kDynThreads) {
    dyn_lv[i] = mono64(i == 0 ? INFINITY : a.pool_logv[base + i]);      // the root ranks first
    newid[i] = -1;
    dep_s[i] = a.pool_depth[base + i];
    par_s[i] = a.pool_parent[base + i];
  }
  __syncthreads();
  for (int i = tid; i < n; i += kDynThreads)
    sel[i] = (i == 0 || (dyn_lv[i] != mono64(-INFINITY) && rank_desc(dyn_lv, n, i) < a.m)) ? 1 : 0;
  if (tid == 0) { count = 1; newid[0] = 0; }
  __syncthreads();
  // the selected entries, compacted (order irrelevant); at most m of them
  int* lst = reinterpret_cast<int*>(dyn_lv);        // the keys are no longer needed
  int* lkey = lst + a.used;
  __shared__ int nsel;
  if (tid == 0) nsel = 0;
  __syncthreads();
  for (int i = 1 + tid; i < n; i += kDynThreads)
    if (sel[i]) lst[atomicAdd(&nsel, 1)] = i;
  __syncthreads();
  const int ns = nsel;
  // breadth-first numbering: a level is ordered by (new id of the parent, pool index), one key per entry of the
  // level (the largest for entries of other levels), so that a place is a count over one array.  An entry whose parent
  // has no id (in a pool where a child outranks its parent) gets none either.
  for (int dep = 1; dep <= a.max_depth; ++dep) {
    if (tid == 0) level_n = 0;
    const int start = count;
    for (int t = tid; t < ns; t += kDynThreads) {
      const int i = lst[t];
      const int pi = dep_s[i] == dep && static_cast<unsigned>(par_s[i]) < static_cast<unsigned>(n) ? newid[par_s[i]] : -1;
      lkey[t] = pi >= 0 ? pi * kDynMaxPool + i : 0x7fffffff;      // (an id is below kDynMaxPool)
    }
    __syncthreads();
    for (int t = tid; t < ns; t += kDynThreads) {
      const int key = lkey[t];
      if (key == 0x7fffffff) continue;
      int pos = 0;
#pragma unroll 8
      for (int t2 = 0; t2 < ns; ++t2) pos += lkey[t2] < key ? 1 : 0;
      const int i = lst[t], id = start + pos;
      const long long o = static_cast<long long>(b) * a.m + id;
      a.parent[o] = key / kDynMaxPool;
      a.token[o] = a.pool_token[base + i];
      a.pool_index[o] = i;
      a.logv[o] = a.pool_logv[base + i];
      newid[i] = id;                                 // read from the next level on
      atomicAdd(&level_n, 1);
    }
    __syncthreads();
    if (tid == 0) count = start + level_n;
    __syncthreads();
  }
  if (tid == 0) {
    const long long o = static_cast<long long>(b) * a.m;
    a.parent[o] = -1; a.token[o] = -1; a.pool_index[o] = 0; a.logv[o] = 0.0;
    a.n_nodes[b] = count;
  }
  for (int i = count + tid; i < a.m; i += kDynThreads) {       // unused tail of the outputs
    const long long o = static_cast<long long>(b) * a.m + i;
    a.parent[o] = -1; a.token[o] = -1; a.pool_index[o] = -1; a.logv[o] = -INFINITY;
  }
}

}  // namespace lantern

namespace lantern {
template <typename T, bool CFG, bool TAU1>
static cudaError_t launch_expand(const ExpandArgs& a, int cs, cudaStream_t st) {
  auto kern = expand_rows_kernel<T, CFG, TAU1>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(expand_smem()));
  if (e != cudaSuccess) return e;
  return launch_after_previous(kern, static_cast<unsigned>(a.B) * a.F * cs, kDynThreads, expand_smem(), st, cs, a);
}
}  // namespace lantern

using namespace lantern;

extern "C" lantern_status lantern_expand_frontier(const lantern_params* p, const void* draft_cond, const void* draft_uncond,
                                                  lantern_dtype dt, int64_t row_stride, int64_t seq_stride, int32_t batch,
                                                  int32_t n_frontier, int32_t n_children, int32_t n_expand,
                                                  const int32_t* frontier, int32_t pool_size, int32_t pool_offset,
                                                  int32_t depth, int32_t* pool_parent, int32_t* pool_token,
                                                  double* pool_logv, int32_t* pool_depth, int32_t* next_frontier,
                                                  void* stream) {
  if (!p || !draft_cond || !frontier || !pool_parent || !pool_token || !pool_logv || !pool_depth || !next_frontier)
    return LANTERN_ERR_INVALID_ARG;
  if (dt != LANTERN_F32 && dt != LANTERN_BF16) return LANTERN_ERR_INVALID_ARG;
  if (batch <= 0 || n_frontier <= 0 || p->vocab <= 0 || !(p->temperature > 0.f) || depth < 1) return LANTERN_ERR_INVALID_ARG;
  if (n_children < 1 || n_children > LANTERN_MAX_CHILDREN || n_expand < 1) return LANTERN_ERR_INVALID_ARG;
  if (p->top_k_draft != 0) return LANTERN_ERR_UNSUPPORTED;          // confidences of truncated rows: not built
  const long long T = static_cast<long long>(n_frontier) * n_children;
  if (T > kDynMaxPool || pool_size > kDynMaxPool) return LANTERN_ERR_UNSUPPORTED;
  if (pool_offset < 1 || pool_offset + T > pool_size) return LANTERN_ERR_INVALID_ARG;
  const int V = p->vocab, lo = p->allowed_begin, hi = p->allowed_end == 0 ? V : p->allowed_end;
  if (lo < 0 || hi > V || lo >= hi) return LANTERN_ERR_INVALID_ARG;
  if (row_stride < V || seq_stride < 0) return LANTERN_ERR_INVALID_ARG;
  ExpandArgs a;
  a.dc = draft_cond; a.du = draft_uncond; a.row_stride = row_stride; a.seq_stride = seq_stride;
  a.B = batch; a.F = n_frontier; a.K = n_children; a.E = n_expand; a.V = V; a.allow_lo = lo; a.allow_hi = hi;
  a.g = p->cfg_scale; a.inv_tau = 1.0f / p->temperature;
  a.frontier = frontier; a.P = pool_size; a.pool_off = pool_offset; a.depth = depth;
  a.pool_parent = pool_parent; a.pool_token = pool_token; a.pool_depth = pool_depth; a.pool_logv = pool_logv;
  a.next_frontier = next_frontier;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const bool cfg = draft_uncond != nullptr, f32 = dt == LANTERN_F32;
  const long long rows = static_cast<long long>(batch) * n_frontier;
  // CTAs per row, as for the draft sampler: every SM a CTA, every warp at least one full step of the row
  int dev = 0, sms = 0, cs = 1;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
    sms = 148;
  const int nvec = (hi - lo) / (f32 ? 4 : 8);
  while (cs < 8 && rows * cs < sms && nvec / (2 * cs * stream::SW) >= 32) cs *= 2;
  if (rows * cs > 0x7fffffffll) return LANTERN_ERR_UNSUPPORTED;
  const bool tau1 = a.inv_tau == 1.0f;
  cudaError_t e;
  if (f32)
    e = cfg ? launch_expand<float, true, false>(a, cs, st)
            : (tau1 ? launch_expand<float, false, true>(a, cs, st) : launch_expand<float, false, false>(a, cs, st));
  else
    e = cfg ? launch_expand<__nv_bfloat16, true, false>(a, cs, st)
            : (tau1 ? launch_expand<__nv_bfloat16, false, true>(a, cs, st) : launch_expand<__nv_bfloat16, false, false>(a, cs, st));
  if (e != cudaSuccess) return LANTERN_ERR_CUDA;
  e = launch_after_previous(select_frontier_kernel, static_cast<unsigned>(batch), kDynThreads, static_cast<size_t>(T) * sizeof(double), st, 1, a);
  return e == cudaSuccess ? LANTERN_OK : LANTERN_ERR_CUDA;
}

extern "C" lantern_status lantern_trim_tree(int32_t batch, int32_t pool_size, int32_t pool_used, int32_t max_depth,
                                            const int32_t* pool_parent, const int32_t* pool_token, const double* pool_logv,
                                            const int32_t* pool_depth, int32_t max_nodes, int32_t* n_nodes, int32_t* parent,
                                            int32_t* token, int32_t* pool_index, double* logv, void* stream) {
  if (!pool_parent || !pool_token || !pool_logv || !pool_depth || !n_nodes || !parent || !token || !pool_index || !logv)
    return LANTERN_ERR_INVALID_ARG;
  if (batch <= 0 || pool_used < 1 || pool_used > pool_size || max_nodes < 1 || max_depth < 0) return LANTERN_ERR_INVALID_ARG;
  if (pool_size > kDynMaxPool || max_nodes > LANTERN_MAX_NODES) return LANTERN_ERR_UNSUPPORTED;
  TrimArgs a;
  a.B = batch; a.P = pool_size; a.used = pool_used; a.m = max_nodes; a.max_depth = max_depth;
  a.pool_parent = pool_parent; a.pool_token = pool_token; a.pool_depth = pool_depth; a.pool_logv = pool_logv;
  a.n_nodes = n_nodes; a.parent = parent; a.token = token; a.pool_index = pool_index; a.logv = logv;
  // (a full pool's 48 KB and the kernel's few static bytes are more than a launch gets unasked)
  const size_t smem = static_cast<size_t>(pool_used) * 24;
  if (smem > 40 * 1024 &&
      cudaFuncSetAttribute(trim_tree_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynMaxPool * 24) != cudaSuccess)
    return LANTERN_ERR_CUDA;
  return launch_after_previous(trim_tree_kernel, static_cast<unsigned>(batch), kDynThreads, smem, static_cast<cudaStream_t>(stream),
                               1, a) == cudaSuccess ? LANTERN_OK : LANTERN_ERR_CUDA;
}
