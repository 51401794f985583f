// Relaxed tree verification for wide rows that are truncated to their top-k entries: the lists come from topk_wide.cuh,
// the per-node part is the one of verify_sparse.cuh.  Two CTAs share an SM, so one node's streaming overlaps the
// other node's on-chip phases.
#pragma once

#include "topk_wide.cuh"

namespace lantern {
namespace wide {

__host__ __device__ constexpr size_t smem_bytes(int V, int cap, int max_children, int kpad) {
  return static_cast<size_t>(region_floats(cap)) * 4 + static_cast<size_t>(4) * cap * 4 + static_cast<size_t>(bins_words(V)) * 4 +
         static_cast<size_t>(2) * bitmap_words(V) * 4 + kCand * 4 + 2 * SW * 2 * 4 + SW * 4 + kMisc * 4 + 16 +
         static_cast<size_t>(max_children) * kpad * 4;
}

// One CTA of 512 threads per node does everything (both rows, then the per-node part); `cap` list entries per side.
// `redo[b*N + n]` is set to 1 when node (b, n) has to be processed by the dense kernel instead, else to 0.
template <typename T, bool CFG>
__global__ void __launch_bounds__(ST, 2) verify_wide_kernel(const VerifyArgs a, int32_t* __restrict__ redo, const int chunk, const int cap) {
  grid_dependency_sync();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using IO = stream::RowIO<T, CFG, false>;
  const int words = bitmap_words(a.V);
  Smem s;
  s.rz = reinterpret_cast<float*>(smem_raw);
  s.rt = reinterpret_cast<int*>(s.rz + kRaw);
  int* ltok[2];                                 // [cap] per side: token, value
  float* lval[2];
  ltok[0] = reinterpret_cast<int*>(s.rz + region_floats(cap));
  lval[0] = reinterpret_cast<float*>(ltok[0] + cap);
  ltok[1] = reinterpret_cast<int*>(lval[0] + cap);
  lval[1] = reinterpret_cast<float*>(ltok[1] + cap);
  s.bins = reinterpret_cast<uint32_t*>(lval[1] + cap);
  uint32_t* bm[2];                              // [words] support bitmaps of the two lists
  bm[0] = s.bins + bins_words(a.V);
  bm[1] = bm[0] + words;
  s.cand = reinterpret_cast<float*>(bm[1] + words);
  Ctx c;
  c.red = s.cand + kCand;
  c.last_red = c.red;
  c.parity = 0;
  s.wtot = reinterpret_cast<uint32_t*>(c.red + 2 * SW * 2);
  s.misc = reinterpret_cast<int*>(s.wtot + SW);
  sparse::NodeSmem ns;
  ns.ut = nullptr;
  ns.uq = s.rz;                                 // the union arrays take over the region of the sample and the raw list
  ns.up = ns.uq + 2 * cap;
  ns.words = words;
  ns.bm[0] = bm[0];
  ns.bm[1] = bm[1];
  ns.rk = s.bins;                               // the histogram is done with by then
  ns.wtot = s.wtot;
  ns.misc = s.misc;
  ns.mbar = reinterpret_cast<uint64_t*>(s.misc + kMisc);
  ns.nbr_s = reinterpret_cast<int*>(ns.mbar + 2);

  const int tid = threadIdx.x;
  if (blockIdx.x == 0 && tid == 0 && a.done) *a.done = 0;      // counter of the repair launch that follows
  // Launch order: blocks of `chunk` CTAs (one per SM) alternate between internal nodes (two rows,
  // sibling loop) and leaves (one row), so that the two CTAs sharing an SM start in different
  // phases and one's streaming overlaps the other's on-chip work.  The grid is padded to whole
  // blocks; CTAs beyond the last node of their kind leave at once.
  int idx;
  {
    const int nI = a.B * a.n_internal, nL = a.B * (a.N - a.n_internal);
    const int mI = (nI + chunk - 1) / chunk, mL = (nL + chunk - 1) / chunk;
    const int cb = blockIdx.x / chunk, off = blockIdx.x - cb * chunk;
    const int both = 2 * min(mI, mL);
    int kind, k;
    if (cb < both) {
      kind = cb & 1;
      k = (cb >> 1) * chunk + off;
    } else {
      kind = mI > mL ? 0 : 1;
      k = (min(mI, mL) + (cb - both)) * chunk + off;
    }
    if (k >= (kind ? nL : nI)) return;
    idx = kind ? nI + k : k;            // position in the internal-first node order
  }
  sparse::NodeId id;
  id.b = idx % a.B;
  id.n = a.order[idx / a.B];
  id.fc = a.first_child[id.n];
  id.nc = a.n_child[id.n];
  id.out_b = static_cast<long long>(id.b) * a.N;
  id.tok_b = a.tokens + id.out_b;
  const long long row_off = static_cast<long long>(id.b) * a.seq_stride + static_cast<long long>(id.n) * a.row_stride;

  const bool bulk_issued = sparse::node_prologue<ST>(a, ns, id);
  for (int w = tid; w < 2 * words; w += ST) bm[0][w] = 0;

  // ---- both rows, one after the other
  const stream::Geo ge = row_geo<IO::VN>(a.allow_lo, a.allow_hi);
  const int nside = id.nc > 0 ? 2 : 1;
  int n_list[2] = {0, 0};
  bool ok = true;
  for (int side = 0; side < nside && ok; ++side) {
    IO io;
    io.c = static_cast<const T*>(side ? a.dc : a.tc) + row_off;
    io.u = CFG ? static_cast<const T*>(side ? a.du : a.tu) + row_off : nullptr;
    io.g = a.g; io.it = a.inv_tau; io.j0 = ge.j0;
    const int kth = side ? a.topk_d : a.topk_t;
    float mx = 0.f, theta = 0.f;
    // the side's list, 2^((z - max) log2 e) per survivor, and its bitmap
    {
      int n_raw = 0;
      ok = stream_topk(c, s, io, ge, kth, n_raw, mx, theta);
      if (!ok) break;
      const float c0 = -mx * kLog2e;
      if (tid == 0) s.misc[10] = 0;
      __syncthreads();
      for (int i0 = 0; i0 < n_raw; i0 += ST) {
        const int i = i0 + tid;
        const float z = i < n_raw ? s.rz[i] : -INFINITY;
        const bool keep = i < n_raw && z >= theta;
        const int pos = reserve(keep ? 1 : 0, &s.misc[10]);
        if (keep && pos < cap) {
          const int t = s.rt[i];
          ltok[side][pos] = t;
          lval[side][pos] = ex2_approx(fmaf(z, kLog2e, c0));
          atomicOr(&bm[side][t >> 5], 1u << (t & 31));
        }
      }
      __syncthreads();
      n_list[side] = s.misc[10];
      ok = n_list[side] <= cap;
    }
  }
  if (!ok) {
    // finish the outstanding bulk copy before leaving (bounded), then hand the node over
    if (bulk_issued) mbar_wait_bounded(smem_u32(ns.mbar), 0);
    if (tid == 0) redo[id.out_b + id.n] = 1;
    return;
  }
  sparse::node_tail<ST, true>(a, c, ns, id, bulk_issued, ltok[0], lval[0], n_list[0], ltok[1], lval[1], n_list[1]);
  if (tid == 0) redo[id.out_b + id.n] = 0;
}

}  // namespace wide
}  // namespace lantern
