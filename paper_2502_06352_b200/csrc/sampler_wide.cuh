// Draft sampling (Sec. 2.1) from wide rows that are truncated to their top-k entries: the list comes from topk_wide.cuh,
// the draw is the one of sampler_sparse.cuh.  A parent whose row does not fit gets the marker kRedoToken in its first
// child's token slot; the dense kernel then draws exactly those parents.
#pragma once

#include "sampler_sparse.cuh"
#include "topk_wide.cuh"

namespace lantern {
namespace wide {

__host__ __device__ constexpr size_t sampler_smem_bytes(int V, int cap) {
  return static_cast<size_t>(2) * kRaw * 4 + static_cast<size_t>(3) * cap * 4 + static_cast<size_t>(bins_words(V)) * 4 +
         static_cast<size_t>(bitmap_words(V)) * 4 + kCand * 4 + 2 * SW * 2 * 4 + SW * 4 + kMisc * 4 + sparse::kDrawInts * 4;
}

template <typename T, bool CFG>
__global__ void __launch_bounds__(ST, 2) sample_wide_kernel(const SampleArgs a, const int cap) {
  grid_dependency_sync();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using IO = stream::RowIO<T, CFG, false>;
  const int words = bitmap_words(a.V);
  Smem s;
  s.rz = reinterpret_cast<float*>(smem_raw);
  s.rt = reinterpret_cast<int*>(s.rz + kRaw);
  int* ltok = s.rt + kRaw;                        // [cap] survivors: token, pre-softmax value, key
  float* lval = reinterpret_cast<float*>(ltok + cap);
  float* keys = lval + cap;
  s.bins = reinterpret_cast<uint32_t*>(keys + cap);
  uint32_t* bm = s.bins + bins_words(a.V);        // [words] their bitmap
  s.cand = reinterpret_cast<float*>(bm + words);
  Ctx c;
  c.red = s.cand + kCand;
  c.last_red = c.red;
  c.parity = 0;
  s.wtot = reinterpret_cast<uint32_t*>(c.red + 2 * SW * 2);
  s.misc = reinterpret_cast<int*>(s.wtot + SW);
  float* pk = reinterpret_cast<float*>(s.misc + kMisc);    // [2][2*SW] warps' best key and token, two buffers

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int idx = blockIdx.x, slot = idx / a.B;
  const int b = idx % a.B;
  const int n = a.inlined ? a.p_node[slot] : a.order[a.order_begin + slot];
  const int fc = a.inlined ? a.p_child[slot] : a.first_child[n], nc = a.inlined ? a.p_count[slot] : a.n_child[n];
  const long long row_off = static_cast<long long>(b) * a.seq_stride + static_cast<long long>(n) * a.row_stride;
  const long long out_b = static_cast<long long>(b) * a.N;

  const stream::Geo ge = row_geo<IO::VN>(a.allow_lo, a.allow_hi);
  IO io;
  io.c = static_cast<const T*>(a.dc) + row_off;
  io.u = CFG ? static_cast<const T*>(a.du) + row_off : nullptr;
  io.g = a.g; io.it = a.inv_tau; io.j0 = ge.j0;
  for (int w = tid; w < words; w += ST) bm[w] = 0;
  float mx = 0.f, theta = 0.f;
  int n_list = 0, n_raw = 0;
  bool ok = stream_topk(c, s, io, ge, a.topk_d, n_raw, mx, theta);
  if (ok) {
    // survivors in token order (ranks in their bitmap), so that sums over the list are the same from run to run
    for (int i = tid; i < n_raw; i += ST)
      if (s.rz[i] >= theta) atomicOr(&bm[s.rt[i] >> 5], 1u << (s.rt[i] & 31));
    __syncthreads();
    const int wpt = (words + ST - 1) / ST, w0 = min(tid * wpt, words), w1 = min(w0 + wpt, words);
    uint32_t* rk = s.bins;
    int cnt = 0;
    for (int w = w0; w < w1; ++w) cnt += __popc(bm[w]);
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) s.wtot[warp] = static_cast<uint32_t>(incl);
    __syncthreads();
    int wt = lane < SW ? static_cast<int>(s.wtot[lane]) : 0, wincl = wt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, wincl, o);
      if (lane >= o) wincl += t;
    }
    int base = __shfl_sync(0xffffffffu, wincl - wt, warp) + incl - cnt;
    n_list = __shfl_sync(0xffffffffu, wincl, SW - 1);
    ok = n_list <= cap;
    if (ok) {
      for (int w = w0; w < w1; ++w) {
        rk[w] = static_cast<uint32_t>(base);
        base += __popc(bm[w]);
      }
      __syncthreads();
      for (int i = tid; i < n_raw; i += ST) {
        const float z = s.rz[i];
        if (z >= theta) {
          const int t = s.rt[i], at = static_cast<int>(rk[t >> 5]) + __popc(bm[t >> 5] & ((1u << (t & 31)) - 1u));
          ltok[at] = t;
          lval[at] = z;
        }
      }
      __syncthreads();
    }
  }
  if (!ok) {
    if (tid == 0) a.tokens[out_b + fc] = sparse::kRedoToken;
    return;
  }

  sparse::ListDraw ld;
  ld.tok = ltok; ld.z = lval; ld.keys = keys; ld.pk = pk;
  ld.n = n_list; ld.mx = mx; ld.theta = theta;
  sparse::draw_from_list<(list_cap(kMaxTopK) + ST - 1) / ST>(a, c, ld, b, n, fc, nc);
}

}  // namespace wide
}  // namespace lantern
