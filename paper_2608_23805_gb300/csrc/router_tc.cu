// Router on tcgen05 tensor cores with fp32-exact products: fp32 logits,
// top-k, softmax weights, shared-expert gate and the per-block expert
// histogram.
//
// The router's top-k output is the route event recorded per layer and graph
// evaluation (paper, Sec. "Output-Exact Execution Beyond the Full-Residency
// Envelope").  Readings: weights are the softmax over the selected k logits;
// equal logits rank the lower expert id first.
//
// Exact split: every fp32 weight w equals hi + mid + lo with hi = bf16(w),
// mid = bf16(w - hi), lo = bf16(w - hi - mid) (each difference is exact in
// fp32 and the last remainder has at most 8 significant bits).  The hidden
// rows are bf16, so every product x * plane is exact in fp32 and
// logits = x Wr^T is three bf16 MMAs accumulating in fp32 -- the same value as
// an fp32 GEMM up to accumulation order.
//
// Two kernels:
//  1. router_logits_kernel, one CTA per (128 tokens, CH experts): sixteen
//     warps read the chunk's fp32 weights, split them and write the three
//     planes as swizzled operand tiles; x tiles come by TMA; 12 MMAs per 64 of
//     K; the logits go to global memory, where the next kernel finds them in
//     L2.  A logit is one accumulation chain over K whatever the call's length
//     and cut: a row's route event does not depend on the rows beside it.
//     What bounds it: the operand feed (x tile and weights, 48 KB per 64 of K
//     at CH = 128, at the SM's 64 bytes a cycle from L2) for long calls, and
//     the latency of one CTA's pass over K for short ones (one token: 24 us as
//     4 CTAs of 128 experts, 16 as 32 of 16).  So short calls are cut into
//     smaller expert chunks (router_chunk).
//  2. router_select_kernel, one warp per token: the top k + 1, weights, gap,
//     the 32-token block's expert histogram and the shared-expert gate
//     sigmoid(x . w_sg).  A call of at most kFuseTokens tokens also does the
//     scatter's work here (offsets, permutation, generation re-check, GEMM
//     groups), in the CTA that finishes last.
#include "permute.cuh"

namespace msi {

namespace {

constexpr int kCvtWarps = 16;                      // weight split, then the epilogue
constexpr int kRlThreads = (kCvtWarps + 2) * 32;   // + TMA producer, MMA issuer
constexpr int kXBytes = 128 * 64 * 2;              // x tile (64 of K)

template <int CH>
struct RlCfg {
  static constexpr int kPlane = CH * 128;          // one plane's rows (64 of K)
  static constexpr int kStage = kXBytes + 3 * kPlane;
  static constexpr int kStages = CH == 128 ? 3 : CH == 64 ? 5 : CH == 32 ? 7 : 8;
  static constexpr int kSmem = 1024 + kStages * kStage + 256;
  // the weight warps in groups that take the stages in turn, so that the
  // loads' and the proxy fence's latencies overlap across the groups; a
  // thread holds its group's next stage in registers.  No more groups than
  // stages: a group that has filled stage `it` knows stages up to
  // it - kStages to be consumed, and the next stage it tests must be at most
  // one phase of its barrier beyond that (a parity cannot tell more).
  static constexpr int kGroups = CH == 128 ? 2 : CH == 16 ? 8 : 4;
  static constexpr int kGroupWarps = kCvtWarps / kGroups;
  static constexpr int kVec = CH * 16 / (kGroupWarps * 32);  // 16-byte loads per thread and stage
  static_assert(kGroups <= kStages && kVec * kGroupWarps * 32 == CH * 16, "weight groups");
  static constexpr int kCols = CH <= 32 ? 32 : CH;  // TMEM columns
};

// hi, mid and lo planes of two weights, as packed bf16 pairs
__device__ __forceinline__ void split3(float a, float b, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
  hi = pack_bf16x2(a, b);
  const float a1 = a - bf16_lo(hi), b1 = b - bf16_hi(hi);
  mid = pack_bf16x2(a1, b1);
  lo = pack_bf16x2(a1 - bf16_lo(mid), b1 - bf16_hi(mid));
}

// The weight warps' loop: the chunk's fp32 rows (src: its first row; H apart),
// 64 of K per stage, into the three planes of the stage.  ALIGNED: src is 16-byte aligned.
template <int CH, bool ALIGNED>
__device__ __forceinline__ void split_weights(const float* src, int H, int nstage, uint8_t* smem,
                                              uint64_t* full, uint64_t* empty, volatile int* abort_flag,
                                              long long lim) {
  using C = RlCfg<CH>;
  // thread: 16-byte piece of the rows row + 2 * kGroupWarps * i of the chunk
  const int group = (threadIdx.x >> 5) / C::kGroupWarps;
  const int gt = threadIdx.x - group * C::kGroupWarps * 32;
  const int row = gt >> 4, piece = gt & 15;
  constexpr int kRowStep = 2 * C::kGroupWarps;
  src += (size_t)row * H + piece * 4;
  float4 v[C::kVec];
  auto load = [&](int it) {
#pragma unroll
    for (int i = 0; i < C::kVec; ++i) {
      const float* p = src + (size_t)(kRowStep * i) * H + it * 64;
      v[i] = ALIGNED ? __ldg(reinterpret_cast<const float4*>(p))
                     : make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
    }
  };
  if (group < nstage) load(group);
  for (int it = group; it < nstage; it += C::kGroups) {
    const int s = it % C::kStages;
    if (!mbar_wait_warp(&empty[s], ((it / C::kStages) & 1) ^ 1, abort_flag, lim)) return;
    const uint32_t st = smem_u32(smem + s * C::kStage) + kXBytes;
#pragma unroll
    for (int i = 0; i < C::kVec; ++i) {
      uint2 pl[3];
      split3(v[i].x, v[i].y, pl[0].x, pl[1].x, pl[2].x);
      split3(v[i].z, v[i].w, pl[0].y, pl[1].y, pl[2].y);
      const int r = row + kRowStep * i;
      const uint32_t at = st + r * 128 + (((piece >> 1) ^ (r & 7)) << 4) + (piece & 1) * 8;
#pragma unroll
      for (int plane = 0; plane < 3; ++plane)
        asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(at + plane * C::kPlane), "r"(pl[plane].x),
                     "r"(pl[plane].y)
                     : "memory");
    }
    if (it + C::kGroups < nstage) load(it + C::kGroups);
    fence_proxy_async_smem();  // before the tensor core's (async proxy) reads
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(&full[s]);
  }
}

template <int CH>
__global__ void __launch_bounds__(kRlThreads, 1)
    router_logits_kernel(const __grid_constant__ CUtensorMap tmX, const RouterTcArgs a,
                         const __grid_constant__ TableParams tp) {
  using C = RlCfg<CH>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::kStages * C::kStage);
  uint64_t* empty = full + C::kStages;
  uint64_t* tfull = empty + C::kStages;
  uint64_t* drain = tfull + 1;
  uint64_t* never = drain + 1;  // no thread ever arrives here
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(never + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // the chunks of one token tile are neighbours in launch order, so the x
  // tile is read from HBM once and from L2 by the other chunks
  const int c = blockIdx.x % a.nchunk;
  const int m0 = a.t0 + blockIdx.x / a.nchunk * 128;
  const int nstage = a.H / 64;
  const long long lim = a.wait_limit;

  if (tid == 0) {
    for (int s = 0; s < C::kStages; ++s) {
      mbar_init(&full[s], 1 + C::kGroupWarps);
      mbar_init(&empty[s], 1);
    }
    mbar_init(tfull, 1);
    mbar_init(drain, 1);
    mbar_init(never, 1);
    *abort_flag = 0;
    mbar_fence_init();
    // the forward's first kernel begins it (status null: a prediction pass,
    // or a later row chunk)
    if (blockIdx.x == 0 && a.begin) {
      forward_begin(a.status, a.sh, a.sh_total, a.T, tp.shared_slot);
      *a.ticket = 0;
    }
  }
  // the resident call's table, copied to global memory for the generation
  // re-check: the entries are read through many SMs' constant caches at once
  if (warp == kCvtWarps && a.begin)
    for (int g = blockIdx.x * 32 + lane; g < tp.E; g += gridDim.x * 32) {
      a.tab_slot[g] = tp.slot[g];
      a.tab_expected[g] = tp.expected[g];
    }
  if (warp == kCvtWarps + 1) {
    tmem_alloc(tmem_slot, C::kCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  grid_release();
  if (warp == kCvtWarps) {
    // ------------------------------------------------------------- x tiles (TMA)
    if (lane == 0) {
      int it = 0;
      for (; it < nstage; ++it) {
        const int s = it % C::kStages;
        if (!mbar_wait(&empty[s], ((it / C::kStages) & 1) ^ 1, abort_flag, lim)) break;
        mbar_arrive_expect_tx(&full[s], kXBytes);
        tma_load_2d(smem + s * C::kStage, &tmX, &full[s], it * 64, m0);
      }
      // on abort the armed loads land before shared memory is released (a
      // stage's barrier may still lack the weight arrivals: bounded)
      if (*abort_flag) {
        for (int d = 0; d < C::kStages && it - 1 - d >= 0; ++d) {
          const int j = it - 1 - d;
          const long long t0 = clock64();
          while (!mbar_try_wait(&full[j % C::kStages], (j / C::kStages) & 1) && clock64() - t0 < kDrainCycles) {
          }
        }
      }
    }
  } else if (warp == kCvtWarps + 1) {
    // ------------------------------------------------------------- MMA issuer
    // (all lanes wait, one elected lane issues)
    bool ok = true;
    const uint32_t tm = uniform(tmem_base);
    uint32_t s = 0, ph = 0;
    for (int it = 0; it < nstage; ++it) {
      ok = mbar_wait_warp(&full[s], ph, abort_flag, lim);
      if (!ok) break;
      tc_fence_after();
      const uint32_t st = smem_u32(smem + s * C::kStage);
      const uint64_t ad = sw128_desc(st);
      if (elect_one()) {
#pragma unroll
        for (int plane = 0; plane < 3; ++plane) {
          const uint64_t bd = sw128_desc(st + kXBytes + plane * C::kPlane);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            umma_bf16(tm, ad + 2 * kk, bd + 2 * kk, idesc_bf16(128, CH), (it | plane | kk) != 0);
        }
        umma_commit(&empty[s]);
      }
      __syncwarp();
      if (++s == C::kStages) {
        s = 0;
        ph ^= 1;
      }
    }
    __syncwarp();
    if (elect_one()) {
      if (ok) umma_commit(tfull);
      umma_commit(drain);
      const long long t0 = clock64();
      while (!mbar_try_wait(drain, 0) && clock64() - t0 < kDrainCycles) {
      }
    }
  } else {
    // ------------------------------------------------------------- weights
    const float* src = a.wr + (size_t)c * CH * a.H;
    if ((reinterpret_cast<uintptr_t>(a.wr) & 15) == 0)
      split_weights<CH, true>(src, a.H, nstage, smem, full, empty, abort_flag, lim);
    else
      split_weights<CH, false>(src, a.H, nstage, smem, full, empty, abort_flag, lim);
    // ------------------------------------------------------------- logits out
    if (a.stall && tid == 0) mbar_wait(never, 0, abort_flag, lim);  // runs out: abort
    const bool ready = __all_sync(0xffffffffu, mbar_wait(tfull, 0, abort_flag, lim)) && !*abort_flag;
    tc_fence_after();
    const int t = m0 + (warp & 3) * 32 + lane;  // TMEM lane: the token
    // the four warps of a lane quarter share the columns, 16 at least each
    constexpr int kPer = CH >= 64 ? CH / 4 : 16;
    const int c0 = (warp >> 2) * kPer;
    if (ready && c0 < CH) {
      const uint32_t tb = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + c0;
      float* dst = a.logits + (size_t)(t - a.t0) * a.E + c * CH + c0;
#pragma unroll
      for (int e0 = 0; e0 < kPer; e0 += 16) {
        uint32_t r[16];
        tmem_ld16(tb + e0, r);
        tmem_ld_wait(r);
        if (t < a.T && t < a.t0 + a.rows) {
          st_global_v8(dst + e0, r);
          st_global_v8(dst + e0 + 8, r + 8);
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == kCvtWarps + 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, C::kCols);
  }
  if (tid == 0 && *abort_flag) atomicCAS(a.status, 0, (int)MSI_ERR_TIMEOUT);
}

// Selection order of the route event: logit descending, then expert id
// ascending.  A logit maps to a 32-bit key with the same order (-0 counted as
// +0; never 0, which stands for no entry); the key above the complement of the
// id is a 64-bit word that is larger the earlier its entry is selected, and no
// two entries share one.
__device__ __forceinline__ uint32_t logit_key(float v) {
  const int b = __float_as_int(v + 0.0f);
  return max((uint32_t)(b ^ ((b >> 31) | (int)0x80000000)), 1u);
}
__device__ __forceinline__ float key_logit(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}
__device__ __forceinline__ unsigned long long entry_word(uint32_t key, int id) {
  return ((unsigned long long)key << 32) | (uint32_t)~id;
}

constexpr int kCand = 64;  // candidates ranked together
struct SelectScratch {     // shared memory of one warp
  uint4 head[8];
  unsigned long long word[kCand];
  unsigned long long best[32];
  int id[kCand];
};

// One warp, one token: ids, weights and gap of token t; returns lane j's
// selected id (j < k).  Lane l holds the experts 128 i + 4 l + c (c < 4,
// i < NV).  The (k + 1)-th largest of the 32 lanes' best logits bounds the
// (k + 1)-th largest of all from below, so the selection is among the entries
// not below it: usually a few more than k + 1.  Each of those finds its rank
// by counting the larger ones.  Every step is a handful of independent
// compares, where k + 1 rounds of a warp argmax are one dependent chain; the
// kernel is bound by its instructions, and by their latency for few tokens.
template <int NV>
__device__ __forceinline__ int select_token(const RouterTcArgs& a, int t, int lane, SelectScratch& sc) {
  const int E = a.E, k = a.k;
  const float* L = a.logits + (size_t)(t - a.t0) * E;
  float4 v[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i)
    v[i] = 128 * i + 4 * lane < E ? *reinterpret_cast<const float4*>(L + 128 * i + 4 * lane)
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
  uint32_t key[4 * NV], hk = 0u;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const bool in = 128 * i + 4 * lane < E;
    const float w[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      key[4 * i + c] = in ? logit_key(w[c]) : 0u;
      hk = max(hk, key[4 * i + c]);
    }
  }
  const int rounds = min(k + 1, E);
  __syncwarp();  // the previous token's readers are done
  reinterpret_cast<uint32_t*>(sc.head)[lane] = hk;
  __syncwarp();
  int above = 0;  // lanes whose best is larger
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint4 q = sc.head[j];
    above += (q.x > hk) + (q.y > hk) + (q.z > hk) + (q.w > hk);
  }
  // at least min(rounds, 32) lanes hold an entry not below the bound, or all
  // lanes with entries do
  const uint32_t bound = max(__reduce_min_sync(0xffffffffu, above < rounds ? hk : 0xFFFFFFFFu), 1u);
  uint32_t mask = 0u;
#pragma unroll
  for (int j = 0; j < 4 * NV; ++j) mask |= key[j] >= bound ? 1u << j : 0u;
  int at = __popc(mask);
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int o = __shfl_up_sync(0xffffffffu, at, off);
    if (lane >= off) at += o;
  }
  const int n = __shfl_sync(0xffffffffu, at, 31);
  at -= __popc(mask);
  if (n <= kCand) {
    for (; mask != 0u; mask &= mask - 1u) {
      const int j = __ffs(mask) - 1;
      sc.id[at++] = 128 * (j >> 2) + 4 * lane + (j & 3);
    }
    __syncwarp();
#pragma unroll 1
    for (int u = 0; u < n; u += 32) {
      const int q = u + lane;
      if (q < n) {
        const int e = sc.id[q];
        sc.word[q] = entry_word(logit_key(L[e]), e);
      }
    }
    __syncwarp();
#pragma unroll 1
    for (int u = 0; u < n; u += 32) {
      const unsigned long long c = u + lane < n ? sc.word[u + lane] : 0ull;
      int r = 0;
#pragma unroll 4
      for (int j = 0; j < n; ++j) r += sc.word[j] > c;
      if (u + lane < n && r < rounds) sc.best[r] = c;
    }
  } else {
    // many entries share few lanes, or one logit: a warp argmax per round
    unsigned long long last = ~0ull;
#pragma unroll 1
    for (int r = 0; r < rounds; ++r) {
      unsigned long long b = 0ull;
#pragma unroll
      for (int j = 0; j < 4 * NV; ++j) {
        const unsigned long long w = entry_word(key[j], 128 * (j >> 2) + 4 * lane + (j & 3));
        if (key[j] != 0u && w < last && w > b) b = w;
      }
#pragma unroll 1
      for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, b, off);
        b = o > b ? o : b;
      }
      if (lane == 0) sc.best[r] = b;
      last = b;
    }
  }
  __syncwarp();
  const unsigned long long mine = sc.best[min(lane, rounds - 1)];
  const int my_i = (int)~(uint32_t)mine;
  const float my_v = key_logit((uint32_t)(mine >> 32));
  const float l0 = __shfl_sync(0xffffffffu, my_v, 0);
  const float ex = lane < k ? expf(my_v - l0) : 0.f;
  float sum = ex;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
  const float lk = __shfl_sync(0xffffffffu, my_v, k - 1);
  const float lk1 = __shfl_sync(0xffffffffu, my_v, k);
  if (lane < k) {
    a.ids[(size_t)t * k + lane] = my_i;
    a.weights[(size_t)t * k + lane] = ex / sum;
  }
  if (a.gap != nullptr && lane == 0) a.gap[t] = (k < E) ? (lk - lk1) : INFINITY;
  return my_i;
}

// sigmoid(x[t] . w_sg) by one warp
__device__ __forceinline__ void shared_gate(const RouterTcArgs& a, int t, int lane) {
  float s = 0.f;
#pragma unroll 4
  for (int h = lane * 8; h < a.H; h += 256) {
    const float4 w0 = __ldg(reinterpret_cast<const float4*>(a.wsg + h));
    const float4 w1 = __ldg(reinterpret_cast<const float4*>(a.wsg + h + 4));
    const uint4 xv = __ldg(reinterpret_cast<const uint4*>(a.x + (size_t)t * a.H + h));
    s = fmaf(bf16_lo(xv.x), w0.x, s);
    s = fmaf(bf16_hi(xv.x), w0.y, s);
    s = fmaf(bf16_lo(xv.y), w0.z, s);
    s = fmaf(bf16_hi(xv.y), w0.w, s);
    s = fmaf(bf16_lo(xv.z), w1.x, s);
    s = fmaf(bf16_hi(xv.z), w1.y, s);
    s = fmaf(bf16_lo(xv.w), w1.z, s);
    s = fmaf(bf16_hi(xv.w), w1.w, s);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if (lane == 0) a.sg[t] = 1.0f / (1.0f + expf(-s));
}

// One CTA per 32-token block, two tokens a warp; the block's histogram is one
// row of bcount for the permutation.
template <int NV>
__global__ void __launch_bounds__(512, 2) router_select_kernel(const RouterTcArgs a) {
  __shared__ int hist[kMaxExperts];
  __shared__ SelectScratch scratch[16];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int e = threadIdx.x; e < a.E; e += blockDim.x) hist[e] = 0;
  __syncthreads();
  grid_wait();
  grid_release();
#pragma unroll 1
  for (int u = 0; u < 2; ++u) {
    const int t = a.t0 + blockIdx.x * 32 + u * 16 + warp;
    if (t >= a.T) break;
    const int id = select_token<NV>(a, t, lane, scratch[warp]);
    if (lane < a.k) atomicAdd(&hist[id], 1);
    if (a.wsg != nullptr) shared_gate(a, t, lane);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < a.E; e += blockDim.x)
    a.bcount[(size_t)(a.t0 / 32 + blockIdx.x) * a.E + e] = hist[e];
}

// A call of at most kFuseTokens tokens: eight tokens a CTA (selection on eight
// warps, the gates on the other eight), and the CTA that finishes last does
// the scatter's work for the whole call: histogram, permutation, generation
// re-check and GEMM groups.  A token names an expert at most once, so an
// expert's rows are the set bits of its token mask: counts and stable ranks
// are population counts.  Latency is all there is to it: one launch instead
// of two or three, and the slots' words are loaded before the ids are known.
template <int NV>
__global__ void __launch_bounds__(512, 2) router_select_scatter_kernel(const RouterTcArgs a,
                                                                       const ScatterArgs s) {
  constexpr int kTok = 8;
  __shared__ ScatterShared sh;
  __shared__ int s_last;
  __shared__ SelectScratch scratch[kTok];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int e = tid;
  grid_wait();
  grid_release();
  int slot = -1, code = 0;
  if (s.tab_slot != nullptr && e < a.E) {
    slot = s.tab_slot[e];
    code = check_code(s.genwords, slot, s.layer, e, s.tab_expected[e]);
  }
  const int t = blockIdx.x * kTok + (warp & (kTok - 1));
  if (t < a.T) {
    if (warp < kTok) select_token<NV>(a, t, lane, scratch[warp]);
    else if (a.wsg != nullptr) shared_gate(a, t, lane);
  }
  if (gridDim.x > 1) {
    __threadfence();  // the ids, before the ticket
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(s.ticket, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
  } else {
    __syncthreads();
  }
  scatter_call(a.ids, a.T, a.k, a.E, s, s.tab_slot != nullptr, slot, code, sh);
}

template <int CH>
cudaError_t launch_logits(const CUtensorMap& tmX, const RouterTcArgs& a, const TableParams& tp, cudaStream_t s) {
  static std::atomic<unsigned long long> attr_done{0};
  constexpr int smem = RlCfg<CH>::kSmem;
  cudaError_t e = smem_attr_once(router_logits_kernel<CH>, smem, attr_done);
  if (e != cudaSuccess) return e;
  const unsigned grid = (unsigned)((a.rows + 127) / 128) * a.nchunk;
  router_logits_kernel<CH><<<grid, kRlThreads, smem, s>>>(tmX, a, tp);
  return cudaGetLastError();
}

template <int NV>
cudaError_t select_nv(const RouterTcArgs& a, const ScatterArgs* sa, cudaStream_t s) {
  if (sa != nullptr) return launch_after(true, router_select_scatter_kernel<NV>, (a.T + 7) / 8, 512, 0, s, a, *sa);
  return launch_after(true, router_select_kernel<NV>, (a.rows + 31) / 32, 512, 0, s, a);
}

}  // namespace

// Experts per logits CTA of a call of T rows: the cut with the least time by a
// fit of the measured launches (event-timed over 1 to 8,192 rows, 512 experts,
// H 2,048, every chunk): about 6 us a CTA, then 0.25 us + 2 ns per expert of
// its chunk for each 64 of K, per round of CTAs on the SMs.
int router_chunk(int T, int E, int sms) {
  const int mt = (T + 127) / 128;
  int best = 16;
  double cost = 1e30;
  for (int ch = 16; ch <= 128 && E % ch == 0; ch *= 2) {
    const int waves = (int)(((long long)mt * (E / ch) + sms - 1) / sms);
    const double c = waves * (6.0 + 32.0 * (0.25 + ch * 0.002));
    if (c < cost) {
      cost = c;
      best = ch;
    }
  }
  return best;
}

cudaError_t launch_router_logits(const CUtensorMap& tmX, const RouterTcArgs& a, const TableParams& tp,
                                 cudaStream_t s) {
  switch (a.chunk) {
    case 16: return launch_logits<16>(tmX, a, tp, s);
    case 32: return launch_logits<32>(tmX, a, tp, s);
    case 64: return launch_logits<64>(tmX, a, tp, s);
    default: return launch_logits<128>(tmX, a, tp, s);
  }
}

cudaError_t launch_router_select(const RouterTcArgs& a, const ScatterArgs* sa, cudaStream_t s) {
  const int nv = (a.E + 127) / 128;
  if (nv <= 1) return select_nv<1>(a, sa, s);
  if (nv <= 2) return select_nv<2>(a, sa, s);
  return select_nv<4>(a, sa, s);
}

}  // namespace msi
