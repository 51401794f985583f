// Stochastic static-tree drafting (Sec. 2.1) for rows that no top-k truncates: streaming kernel.
//
// The s children of a parent are the s largest keys z_j + G_j, G_j = -log(-log U_j) (Gumbel-top-s,
// sampling without replacement from p).  The drafter row is streamed from HBM once and never held
// on chip.  The first chunk's elements get float32 keys from fast logarithms (absolute error below
// kKeyEps); the (s+4)-th best of a few of them is a threshold T.  Every later element only has to
// show whether it could beat T: z + G > T means -log U < e^(z-T), and -log U >= 1 - U, so an element
// with 1 - U >= e^(z-T) is out.  That test costs one exponential and no logarithm, and the few
// elements that pass it go to a candidate list in shared memory, whose keys are formed when the list
// is cut back to its s+4 best entries and T rises to the last of them.  Every element left out has
// key <= T.  At the end the few candidates are ranked by their float32 keys, or, when two of them (or
// one and T) are closer than the keys' errors, by keys recomputed in double precision (ties: lower
// token id); the result is the exact ranking as long as the s-th exact key clears T by kKeyEps, which
// is checked (LANTERN_DEV_KEY_TIES otherwise: more than s+4 keys within 2.5e-4 of each other at the
// top, or within a few units in the last place of logits so large that those are more).  The softmax
// denominator for draft_prob comes from the same pass.
//
// Bound: instruction issue; the generator alone is 10 to 12 of about 27 instructions per element.  3200 rows of
// 65536 bfloat16 logits: 244 us (two logarithms per element and branches between the vectors: 320); 144 rows of
// 65536 float32 logits with guidance: 28 us, was 40; a row whose elements are one chunk per CTA is a chain of
// barriers, 8 us on 8 CTAs.
#pragma once
#include "toplist.cuh"

namespace lantern {
namespace stream {

// bound on |fast key - exact key| (up to the constant below): the logarithms' error, and the key's own rounding, which is
// what counts for logits in the thousands and above (2^-24 of the key, doubled)
constexpr float kKeyEps = 2.5e-4f;
__device__ __forceinline__ float key_eps(float k) { return fmaf(fabsf(k), 1.1920929e-7f, kKeyEps); }
constexpr float kKeyShift = -0.36651292f;        // ln(ln 2): fast keys are z + G + ln(ln 2)

__host__ __device__ constexpr size_t sampler_stream_smem() {
  return kSmallBytes + kListCap * 8 + kFinal * 16 + 2 * 2 * SW * 8 + 16 * 8 + kMaxCluster * 8;
}

__device__ __forceinline__ float lg2_approx(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// float32 key of one element: z - ln2 * lg2(-lg2 U) (the constant -ln(ln 2) is the same for all).
// lg2.approx is accurate to 2^-22 absolutely near 1, so for U > 0.999 (where -lg2 U is tiny) the
// callers redo the inner logarithm with logf.
__device__ __forceinline__ float fast_key(float z, float U) {
  return fmaf(-0.6931471805599453f, lg2_approx(-lg2_approx(U)), z);
}
__device__ __noinline__ float careful_key(float z, float U) {
  return fmaf(-0.6931471805599453f, lg2_approx(-logf(U) * kLog2e), z);
}
// ... and where U is below the smallest normal number, which lg2.approx takes for 0 (supplied uniforms only)
__device__ __forceinline__ bool wants_care(float U) { return U > 0.999f || U < 1.17549435e-38f; }

template <typename T, bool CFG, bool TAU1>
__global__ void __launch_bounds__(ST, 4) sample_stream_kernel(const SampleArgs a) {
  grid_dependency_sync();
  using IO = RowIO<T, CFG, TAU1>;
  constexpr int VN = IO::VN;
  constexpr int UV = (CFG ? 2 : 4) * 4 / VN;     // vectors per thread and iteration (ST*UV*VN <= kIterElems)
  static_assert(ST * UV * VN <= kIterElems, "iteration size");
  extern __shared__ __align__(16) unsigned char samp_smem[];
  SCtx c;
  float* small = reinterpret_cast<float*>(samp_smem);
  c.red = small;
  c.xch = c.red + 2 * SW * 4;
  c.gath = c.xch + 8;
  int* misc = reinterpret_cast<int*>(c.gath + kMaxCluster * 4);     // [32]
  TopList s;
  s.list = reinterpret_cast<uint2*>(samp_smem + kSmallBytes);
  s.fin = s.list + kListCap;
  s.fkey = reinterpret_cast<double*>(s.fin + kFinal);
  s.pk = reinterpret_cast<uint2*>(s.fkey + kFinal);
  s.top = s.pk + 2 * 2 * SW;
  s.rinfo = s.top + 16;
  s.cnt = misc;
  c.rank = cluster_ctarank();
  c.nrank = cluster_nctarank();
  c.parity = 0;
  if (c.nrank > 1) cluster_arrive_relaxed();          // waited for before the first access to a peer's shared memory

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int idx = blockIdx.x / c.nrank;
  const int b = idx % a.B, slot = idx / a.B;
  // few parents travel with the launch: no chain of reads in front of the row's first load
  const int n = a.inlined ? a.p_node[slot] : a.order[a.order_begin + slot];
  const int fc = a.inlined ? a.p_child[slot] : a.first_child[n], nc = a.inlined ? a.p_count[slot] : a.n_child[n];
  const long long row_off = static_cast<long long>(b) * a.seq_stride + static_cast<long long>(n) * a.row_stride;
  const long long out_b = static_cast<long long>(b) * a.N;
  const uint32_t row_id = static_cast<uint32_t>(out_b + n);
  const float* gum = a.gumbel ? a.gumbel + static_cast<long long>(row_id) * a.V : nullptr;
  const bool want_prob = a.draft_prob != nullptr;
  const int R = nc + kExtra;

  Geo ge;
  ge.alo = a.allow_lo; ge.ahi = a.allow_hi;
  ge.j0 = ge.alo / VN * VN;
  ge.nvec = (ge.ahi - ge.j0 + VN - 1) / VN;
  ge.vi0 = ge.alo > ge.j0 ? 1 : 0;
  ge.vi1 = (ge.j0 + ge.nvec * VN > ge.ahi) ? ge.nvec - 1 : ge.nvec;
  if (ge.vi1 < ge.vi0) ge.vi1 = ge.vi0;
  const int nwarps = static_cast<int>(c.nrank) * SW;
  ge.vw = ((ge.nvec + nwarps - 1) / nwarps + 31) / 32 * 32;
  const int gw = static_cast<int>(c.rank) * SW + warp;
  const int vbeg = min(gw * ge.vw, ge.nvec), vend = min(vbeg + ge.vw, ge.nvec);

  IO io;
  io.c = static_cast<const T*>(a.dc) + row_off;
  io.u = CFG ? static_cast<const T*>(a.du) + row_off : nullptr;
  io.g = a.g; io.it = a.inv_tau; io.j0 = ge.j0;

  if (tid == 0) *s.cnt = 0;
  __syncthreads();

  // 1 + U of tokens j .. j+VN-1 (j a multiple of VN), to 2^-24: enough for the test of the later chunks.  Philox words
  // become floats without an integer conversion: the 23 mantissa bits under the exponent of 1.0 give F = 1 + i 2^-23, and
  // subtracting 1 - 2^-24 leaves U = (i + 1/2) 2^-23 exactly.  Supplied uniforms lie on no such grid: keys are
  // made from `uniforms`, which hands them on as they are.
  auto words = [&](int j, float (&F)[VN]) {
    if (gum) {
#pragma unroll
      for (int e = 0; e < VN; ++e) F[e] = 1.f + ((j + e < a.V) ? __ldcs(gum + j + e) : 0.5f);
    } else {
#pragma unroll
      for (int q = 0; q < VN / 4; ++q) {
        const Philox4 r = philox4x32_10_keys(static_cast<uint32_t>((j >> 2) + q), row_id, static_cast<uint32_t>(a.step),
                                             (static_cast<uint32_t>(a.step >> 32) << 2) | kStreamGumbel, a.rk0, a.rk1);
        const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) F[4 * q + e] = __uint_as_float(__funnelshift_r(w[e], 0x7fu, 9));
      }
    }
  };
  auto uniforms = [&](int j, float (&U)[VN]) {
    if (gum) {
#pragma unroll
      for (int e = 0; e < VN; ++e) U[e] = (j + e < a.V) ? __ldcs(gum + j + e) : 0.5f;
    } else {
      words(j, U);
#pragma unroll
      for (int e = 0; e < VN; ++e) U[e] -= 0.99999994f;
    }
  };
  auto uniform_at = [&](int t) -> float {
    if (gum) return __ldcs(gum + t);
    const Philox4 r = philox4x32_10_keys(static_cast<uint32_t>(t >> 2), row_id, static_cast<uint32_t>(a.step),
                                         (static_cast<uint32_t>(a.step >> 32) << 2) | kStreamGumbel, a.rk0, a.rk1);
    return uniform_open((t & 3) == 0 ? r.x : ((t & 3) == 1 ? r.y : ((t & 3) == 2 ? r.z : r.w)));
  };
  // Cut of the list to its R best entries; entries from `raw` on still hold z in the place of their key.
  auto cut = [&](int raw, float T) -> float {
    const int n = min(*s.cnt, kListCap);
    for (int i = raw + tid; i < n; i += ST) {
      const uint2 en = s.list[i];
      const float U = uniform_at(static_cast<int>(en.y)), z = __uint_as_float(en.x);
      s.list[i].x = __float_as_uint(wants_care(U) ? careful_key(z, U) : fast_key(z, U));
    }
    __syncthreads();
    return n <= ST ? cut_ranked(s, R, T) : cut_list(s, R, T);
  };

  // One entry for the list (appends are rare after the first cut: a shared-memory atomic each)
  auto append = [&](float k, int tok) {
    const int pos = atomicAdd(s.cnt, 1);
    if (pos < kListCap) s.list[pos] = make_uint2(__float_as_uint(k), static_cast<uint32_t>(tok));
  };
  // Optimistic pass.  The first chunk's keys stay in registers until a first threshold is known: the
  // R-th best of the warps' two best keys each (distinct tokens, so a lower bound of the row's R-th
  // best key), found with one barrier; the chunk's keys above it then enter the list.  One cut of the
  // (short) list after a third of the row tightens the threshold (more cuts cost more in barriers than
  // they save in appends); the other chunks run without barriers.  If the list overflows all the same (keys that keep growing along the row), the
  // row is redone with a check after every chunk.
  float Tk = -INFINITY;                               // every element left out has key <= Tk
  float mx = -INFINITY, sx = 0.f;
  int raw = kListCap;                                 // list entries from here on have no key yet
  const int iters = (ge.vw + 32 * UV - 1) / (32 * UV);
  const int cut_it = max(1, iters / 3);                // the one scheduled cut of the optimistic pass
  for (int mode = 0; mode < 2; ++mode) {
    Tk = -INFINITY;
    mx = -INFINITY;
    sx = 0.f;
    raw = kListCap;
    // ---- first chunk
    {
      uint4 rc[UV], ru[UV];
#pragma unroll
      for (int u = 0; u < UV; ++u) {
        const int vv = vbeg + 32 * u + lane;
        if (vv < vend && vv >= ge.vi0 && vv < ge.vi1) io.load(vv, rc[u], ru[u]);
      }
      float first[UV][VN];                              // keys of the first chunk
      float tbk = -INFINITY;                            // ... and the thread's best of them
      int tbj = 0x7fffffff;
#pragma unroll
      for (int u = 0; u < UV; ++u) {
        const int vv = vbeg + 32 * u + lane;
        const int j = ge.j0 + vv * VN;
        float z[VN];
#pragma unroll
        for (int e = 0; e < VN; ++e) first[u][e] = -INFINITY;
        if (vv < vend) {
          if (vv >= ge.vi0 && vv < ge.vi1) {
            io.z(rc[u], ru[u], z);
          } else {                                      // ragged first / last vector of the row
#pragma unroll
            for (int e = 0; e < VN; ++e) z[e] = (j + e >= ge.alo && j + e < ge.ahi) ? io.z_at(j + e) : -INFINITY;
          }
          float U[VN];
          uniforms(j, U);
          bool care = false;
#pragma unroll
          for (int e = 0; e < VN; ++e) {
            first[u][e] = fast_key(z[e], U[e]);
            care |= wants_care(U[e]);
          }
          if (care) {                                   // rare: one vector in a hundred
#pragma unroll
            for (int e = 0; e < VN; ++e)
              if (wants_care(U[e])) first[u][e] = careful_key(z[e], U[e]);
          }
          if (want_prob) acc_exp<VN>(z, mx, sx);
        }
#pragma unroll
        for (int e = 0; e < VN; ++e)
          if (key_before(first[u][e], j + e, tbk, tbj)) { tbk = first[u][e]; tbj = j + e; }
      }
      Tk = first_threshold(s, R, tbk, tbj);             // (R <= 12 <= 2 * SW)
      // (the key at the threshold itself belongs to the R best: >=, so that the first cut finds R entries)
#pragma unroll
      for (int u = 0; u < UV; ++u) {
        const int j = ge.j0 + (vbeg + 32 * u + lane) * VN;
#pragma unroll
        for (int e = 0; e < VN; ++e)
          if (first[u][e] >= Tk && first[u][e] > -INFINITY) append(first[u][e], j + e);
      }
    }
    if (iters > 1) {
      __syncthreads();
      raw = min(*s.cnt, kListCap);
      __syncthreads();                                  // everyone has read the count before it moves again
      if (mode == 1 && raw > kListCap - kIterElems) {
        Tk = cut(raw, Tk);
        raw = R;
      }
    }
    // ---- the other chunks: an element passes when 1 + U > 2 - e^(z - Tk), with room for the roundings of
    // z L - Tk L (2^-24 of either), of the exponential (2^-22 relative) and of the two sides (2^-24 each)
    auto cutoff = [](float T) { return fmaf(-(T - kKeyShift), kLog2e, fmaf(fabsf(T), 1e-6f, 4e-5f)); };
    float c0 = cutoff(Tk);
    constexpr float kPass = 1.9999995f;
    for (int it = 1; it < iters; ++it) {
      const int base = vbeg + it * 32 * UV;
      uint4 rc[UV], ru[UV];
      if (base >= ge.vi0 && base + 32 * UV <= min(vend, ge.vi1)) {
        // whole vectors only (the same decision in every lane): no branch between the vectors, so that their
        // generator rounds interleave and share the round keys
        float F[UV][VN];
#pragma unroll
        for (int u = 0; u < UV; ++u) io.load(base + 32 * u + lane, rc[u], ru[u]);
#pragma unroll
        for (int u = 0; u < UV; ++u) words(ge.j0 + (base + 32 * u + lane) * VN, F[u]);
#pragma unroll
        for (int u = 0; u < UV; ++u) {
          float z[VN];
          io.z(rc[u], ru[u], z);
          float best = 0.f;
#pragma unroll
          for (int e = 0; e < VN; ++e) {
            F[u][e] += ex2_approx(fmaf(z[e], kLog2e, c0));
            best = fmaxf(best, F[u][e]);
          }
          if (want_prob) acc_exp<VN>(z, mx, sx);
          if (best > kPass) {                           // rare, and rarer after the cut
#pragma unroll
            for (int e = 0; e < VN; ++e)
              if (F[u][e] > kPass && z[e] > -INFINITY) append(z[e], ge.j0 + (base + 32 * u + lane) * VN + e);
          }
        }
      } else {
#pragma unroll 1
        for (int u = 0; u < UV; ++u) {
          const int vv = base + 32 * u + lane;
          const int j = ge.j0 + vv * VN;
          if (vv < vend) {
            float z[VN], F[VN];
            if (vv >= ge.vi0 && vv < ge.vi1) {
              io.load(vv, rc[0], ru[0]);
              io.z(rc[0], ru[0], z);
            } else {                                    // ragged first / last vector of the row
#pragma unroll
              for (int e = 0; e < VN; ++e) z[e] = (j + e >= ge.alo && j + e < ge.ahi) ? io.z_at(j + e) : -INFINITY;
            }
            words(j, F);
#pragma unroll
            for (int e = 0; e < VN; ++e)
              if (F[e] + ex2_approx(fmaf(z[e], kLog2e, c0)) > kPass && z[e] > -INFINITY) append(z[e], j + e);
            if (want_prob) acc_exp<VN>(z, mx, sx);
          }
        }
      }
      if (it == cut_it || mode == 1) {
        __syncthreads();
        const int cn = *s.cnt;
        __syncthreads();                                // everyone has read the count before it moves again
        if (mode == 1 ? cn > kListCap - kIterElems : cn > R) {
          if (cn <= kListCap) {                         // (an overflowing list is redone anyway)
            Tk = cut(raw, Tk);
            raw = min(cn, R);
            c0 = cutoff(Tk);
          }
        }
      }
    }
    __syncthreads();
    const bool overflow = *s.cnt > kListCap;
    if (!overflow) break;
    __syncthreads();                                    // (mode 1 never overflows: it cuts in time)
    if (tid == 0) *s.cnt = 0;
    __syncthreads();
  }
  if (c.nrank > 1) cluster_wait();                      // every CTA of the row has started

  // ---- softmax denominator of the row (for draft_prob)
  float gm[1] = {0.f}, gs[1] = {0.f};
  if (want_prob) {                                    // (uniform: a kernel argument)
    gm[0] = warp_max(mx);
    combine<1, true>(c, gm);
    if (gm[0] == -INFINITY) gm[0] = 0.f;
    gs[0] = warp_sum(mx == -INFINITY ? 0.f : sx * ex2_approx((mx - gm[0]) * kLog2e));
    combine<1, false>(c, gs);
  }

  // ---- every CTA's R best entries in order; those of all CTAs of the row go to CTA 0
  Tk = cut(raw, Tk);
  const int mine = *s.cnt;
  const uint2* fin = s.list;
  int nf = mine;
  float tmax = Tk;
  if (c.nrank > 1) {
    if (tid < mine) dsmem_st_u64(dsmem_addr(smem_u32(&s.fin[c.rank * kMaxR + tid]), 0), s.list[tid]);
    if (tid == 0)
      dsmem_st_u64(dsmem_addr(smem_u32(&s.rinfo[c.rank]), 0), make_uint2(static_cast<uint32_t>(mine), __float_as_uint(Tk)));
    cluster_sync();
    if (c.rank != 0) return;
    for (uint32_t r = 0; r < c.nrank; ++r) tmax = fmaxf(tmax, __uint_as_float(s.rinfo[r].y));
    nf = merge_lists(s, c.nrank);
  }
  // ---- exact order: float32 keys decide unless two neighbours in the order, or the last child and the
  // elements left out, are closer than the keys' errors
  bool near = false;
  if (tid < nf && tid < nc) {
    const float k = __uint_as_float(fin[tid].x);
    if (tid + 1 < nf) {
      const float next = __uint_as_float(fin[tid + 1].x);
      near = k - next <= key_eps(k) + key_eps(next);
    }
    if (tid == nc - 1) near |= tmax > -INFINITY && k - tmax <= key_eps(k) + key_eps(tmax);
  }
  const bool exact = __syncthreads_or(near ? 1 : 0) != 0;
  if (exact && tid < nf)
    s.fkey[tid] = static_cast<double>(io.z_at(static_cast<int>(fin[tid].y))) -
                  log(-log(static_cast<double>(uniform_at(static_cast<int>(fin[tid].y)))));
  if (exact) __syncthreads();
  if (tid < nf) {
    const int t = static_cast<int>(fin[tid].y);
    int rank = tid;
    if (exact) {
      const double k = s.fkey[tid];
      rank = 0;
      for (int i = 0; i < nf; ++i) {
        const double ki = s.fkey[i];
        rank += (ki > k || (ki == k && static_cast<int>(fin[i].y) < t)) ? 1 : 0;
      }
      if (rank == nc - 1 && static_cast<double>(tmax) + key_eps(tmax) >= k + kKeyShift) vflag(a.status, LANTERN_DEV_KEY_TIES);
    }
    if (rank < nc) {
      a.tokens[out_b + fc + rank] = t;
      if (want_prob) {
        const float zt = io.z_at(t);
        a.draft_prob[out_b + fc + rank] = gs[0] > 0.f ? ex2_approx(fmaf(zt, kLog2e, -gm[0] * kLog2e)) / gs[0] : 0.f;
      }
    }
  }
  if (tid >= nf && tid < nc) {                        // fewer than s tokens with positive probability
    a.tokens[out_b + fc + tid] = -1;
    if (want_prob) a.draft_prob[out_b + fc + tid] = 0.f;
  }
  if (nf == 0 && tid == 0) vflag(a.status, LANTERN_DEV_EMPTY_ROW);
}

}  // namespace stream
}  // namespace lantern
