// Device helpers of the kernels that build a call's permutation and GEMM
// groups (permute.cu; the one-CTA selection in router_tc.cu).
#pragma once

#include "kernels.cuh"

namespace msi {

// Generation re-check of one slot (fail closed): 0 or the status to report.
__device__ __forceinline__ int check_code(const GenWord* gw, int slot, int layer, int e,
                                          unsigned long long expected) {
  if (slot < 0) return MSI_ERR_NOT_RESIDENT;
  const unsigned long long obj = gw[slot].obj;
  const unsigned long long gen = gw[slot].gen;
  if (obj != obj_key(layer, e)) return MSI_ERR_WRONG_OBJECT;
  if (gen != expected) return MSI_ERR_STALE_GENERATION;
  return 0;
}

// Exclusive scan of one value per thread over the block (tmp: one word per
// warp); synchronise before tmp is used again.
__device__ __forceinline__ int block_excl_scan(int v, int* tmp, int* total) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int incl = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int o = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += o;
  }
  if (lane == 31) tmp[warp] = incl;
  __syncthreads();
  const int nw = blockDim.x >> 5;
  int base = 0, tot = 0;
  for (int w = 0; w < nw; ++w) {
    if (w < warp) base += tmp[w];
    tot += tmp[w];
  }
  *total = tot;
  return base + incl - v;
}

// Minimum over the block, in every thread.
__device__ __forceinline__ int block_min(int v, int* tmp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, off));
  __syncthreads();
  if (lane == 0) tmp[warp] = v;
  __syncthreads();
  int m = 0x7fffffff;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = min(m, tmp[w]);
  return m;
}

// Resident call, one expert per thread (thread e: expert e of cnt rows from
// permuted row row_begin, in `slot`, code: its generation re-check): the GEMM
// groups with their 128- and 256-row tile prefixes, and the lowest failing
// expert's status.  Every thread of the block calls it.
__device__ __forceinline__ void build_groups(const ScatterArgs& a, int e, int cnt, int row_begin, int slot,
                                             int code, int* tmp) {
  const bool ok = e < a.E && code == 0;
  const int mt = ok ? (cnt + kBM - 1) / kBM : 0, pt = ok ? (cnt + 2 * kBM - 1) / (2 * kBM) : 0;
  int mtot, ptot;
  __syncthreads();
  const int mb = block_excl_scan(mt, tmp, &mtot);
  __syncthreads();
  const int pb = block_excl_scan(pt, tmp, &ptot);
  if (e < a.E) {
    Group g;
    g.row_begin = row_begin;
    g.row_count = cnt;
    g.slot = slot < 0 ? 0 : slot;
    g.mt_begin = mb;
    g.ok = code == 0;
    g.expert = e;
    g.pt_begin = pb;
    g.pad1 = 0;
    a.groups[e] = g;
  }
  const int m = block_min(code ? (e << 4) | code : 0x7fffffff, tmp);
  if (threadIdx.x == 0) {
    a.total_mtiles[0] = mtot;
    a.total_mtiles[1] = ptot;
    if (m != 0x7fffffff) atomicCAS(a.status, 0, m & 15);
  }
}

// The scatter's work for a whole call of at most kFuseTokens tokens, by one
// block of at least kMaxExperts threads once every id is written: offsets,
// counts, permutation and, for a resident call, the generation re-check (slot
// and code of the thread's expert) and the GEMM groups.  A token names an
// expert at most once, so an expert's rows are the set bits of its token mask:
// counts and stable ranks are population counts.
struct ScatterShared {
  unsigned mask[kFuseTokens / 32][kMaxExperts];
  int offs[kMaxExperts];
  int tmp[32];
};
__device__ __forceinline__ void scatter_call(const int* ids, int T, int k, int E, const ScatterArgs& s, bool resident,
                                             int slot, int code, ScatterShared& sh) {
  const int tid = threadIdx.x, e = tid, nw = (T + 31) / 32;
  if (tid < kMaxExperts)
    for (int w = 0; w < nw; ++w) sh.mask[w][tid] = 0u;
  for (int r = tid; r < s.n_ready; r += blockDim.x) s.ready[r] = 0;
  __syncthreads();
  const int n = T * k;
  for (int f = tid; f < n; f += blockDim.x) {
    const int tok = f / k;
    atomicOr(&sh.mask[tok >> 5][__ldcg(&ids[f])], 1u << (tok & 31));
  }
  __syncthreads();
  int cnt = 0;
  if (e < E)
    for (int w = 0; w < nw; ++w) cnt += __popc(sh.mask[w][e]);
  int total;
  const int base = block_excl_scan(cnt, sh.tmp, &total);
  if (e < E) {
    sh.offs[e] = base;
    s.offsets[e] = base;
    s.counts_out[e] = cnt;
  }
  if (tid == 0) s.offsets[E] = total;
  __syncthreads();
  for (int f = tid; f < n; f += blockDim.x) {
    const int tok = f / k, id = __ldcg(&ids[f]), w = tok >> 5;
    int pos = sh.offs[id] + __popc(sh.mask[w][id] & ((1u << (tok & 31)) - 1u));  // + the expert's earlier tokens
    for (int q = 0; q < w; ++q) pos += __popc(sh.mask[q][id]);
    s.perm[pos] = tok;
    s.inv[f] = pos;
  }
  if (resident) build_groups(s, e, cnt, base, slot, cnt > 0 ? code : 0, sh.tmp);
}

}  // namespace msi
