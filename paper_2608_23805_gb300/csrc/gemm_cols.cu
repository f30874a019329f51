// The expert FFN with weights as the MMA's rows and tokens as its columns, in
// one persistent launch (sm_103a).
//
// Each selected expert runs its complete gate, up and down projections
// (paper, Sec. "Output-Exact Execution Beyond the Full-Residency Envelope")
// on weights read from the stable slot address the Plan published for it
// (Sec. "Stable Slots and Bundle Publication").
//
// A tile is 128 weight rows x up to 32, 64 or 128 tokens of one expert (N = the tile's
// tokens rounded up to 16, so an expert's few rows cost their own MMA time
// and not that of 128):
//   up tile (g, m, n):    64 intermediate units, as rows 16 gate, 16 up, 16
//       gate, ... (lanes 16 apart hold gate and up of a unit, one shuffle
//       brings them together): h[rows, 64 n .. 64 n + 64) = silu(g) * u
//   down tile (g, m, n):  128 output features: y[rows, 128 n .. 128 n + 128)
// A short resident call's shared expert is one more group (all tokens, identity
// rows; cols_shared in plan.cu).
//
// K goes by stages of four steps of 64 (two where four would leave too few
// stages), one tcgen05.commit a stage: the issuing and the token warp's
// per-stage instructions, not the MMAs, bound short tiles.
// Weights (operand A):
//   bf16: TMA into the stage, read by the MMA from shared memory;
//   4-bit: TMA brings 128 rows x 256 codes (16 KB) and cp.async their scales
//       into a ring of their own; sixteen warps in four sets (set j: every
//       fourth half stage) convert 128 codes of a row per thread and write them
//       to a TMEM operand ring of two stages, from which the MMA reads A.
//       The weights thus cross shared memory once, as codes: converted in
//       shared memory they would cost 4 x their bf16 size in shared-memory
//       traffic, which bounds the row-major 4-bit kernel.
// Tokens (operand B), in the 128-byte swizzle, the tile's rows only: h by TMA in
// boxes of 16 rows; x through the permutation, by TMA gathers of four rows up to
// 64 tokens a tile, else by cp.async.  Copies and gathers by size (a call with the
// shared expert in the launch, us):
//   tokens               37    250    800   1,600   4,096
//   cp.async, x and h   195    346    382     421     537
//   gathers for x       187    334    369     427     562
//   cp.async for x      -       352    382     406     521
// A gather frees the schedulers that the conversion needs, but brings fewer
// bytes a cycle than 128 threads' copies, which is what counts in large tiles.
//
// What bounds it: for 4-bit the instructions of the converting and the issuing
// warps (an MMA of up to 96 columns takes 48 cycles), not HBM; for bf16 and few
// tokens the latency of a tile's pass over K.  Resident Qwen-shaped layer, both
// projections: 4-bit 250 tokens 271 us (534 as two row-major launches), 4,096
// tokens 393 us (546), 8 tokens 62 us with the shared expert (91 without it);
// bf16 one token 26 us with the shared expert (row-major 28 without it, which
// took 25 beside it).
//
// Schedule: every CTA takes a contiguous range of the up tiles, then of the
// down tiles (ColsWalk), so a role steps from tile to tile without a search.
// A down tile needs its token tile's h rows: per-token-tile counters, released
// by the up epilogue, acquired by the token warps; the weight producer does
// not wait for them and runs ahead into the down tiles' weights.  Every CTA
// runs its up tiles first and the launch is cooperative, so every wait ends;
// every wait is bounded as in the other GEMMs.
//
// Roles: warps 0-3 epilogue, 4 MMA + TMEM, 5 weight producer, 6-9 tokens, and
// 4-bit 10-25 conversion.
#include <cuda_fp16.h>

#include "internal.cuh"

namespace msi {

namespace {

constexpr int kCSlot = 128 * 128;     // weight ring slot
constexpr int kCScale = 128 * 16;     // 4-bit: its rows' eight scales
constexpr int kCRingMax = 8;
constexpr int kCOperand = 4;          // 4-bit: half stages that the TMEM operand ring holds
constexpr int kCTokWarps = 4;
constexpr int kCDqWarp0 = 10;
constexpr int kCDqWarps = 16;
constexpr int kCTable = kMaxExperts + 1;  // groups: experts and the shared one

constexpr uint32_t kCOperandCol = 256;    // TMEM: two accumulators of 128 columns, then A steps
constexpr int cols_threads(bool q4) { return (kCDqWarp0 + (q4 ? kCDqWarps : 0)) * 32; }

// Ring position: slot index and the parity of its round.
struct Ring {
  int n, i = 0;
  uint32_t ph = 0;
  __device__ __forceinline__ explicit Ring(int n_) : n(n_) {}
  __device__ __forceinline__ void step() {
    if (++i == n) {
      i = 0;
      ph ^= 1;
    }
  }
};

__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, uint64_t* bar, int c0, int c1,
                                            int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, "
      "%5, %6}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}

// Four rows of a map whose box is one row of 64: 4 x 128 swizzled bytes.
__device__ __forceinline__ void tma_gather4(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c, int r0, int r1,
                                            int r2, int r3) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes [%0], [%1, {%3, "
      "%4, %5, %6, %7}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c), "r"(r0), "r"(r1), "r"(r2), "r"(r3)
      : "memory");
}

// Generic-proxy writes to global memory (observed through an acquire) before
// this thread's TMA loads of them.
__device__ __forceinline__ void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}

__device__ __forceinline__ void cp_async16_at(uint32_t dst, const void* src, uint32_t src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}

__device__ __forceinline__ uint64_t desc64(uint32_t lo, uint32_t hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(hi));
  return d;
}

// D[tmem] (+)= A[tmem] * B[smem]^T
__device__ __forceinline__ void umma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                             uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// 32 lanes x 16 consecutive 32-bit columns, registers to TMEM
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
      "%13, %14, %15, %16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
      "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ uint32_t fma_bf16x2(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
__device__ __forceinline__ uint32_t mul_bf16x2(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

// Eight 4-bit codes -> eight bf16 weights s (q - 8), each rounded once (the
// bits of dequant8), in packed bf16 arithmetic: 33 cycles a word and scheduler
// against 36, and seven instead of fifteen on the ALU pipe that the rest of
// the kernel needs (250 tokens: 308 us, with dequant8 318).  A code as the low bits of a
// bf16 is the subnormal q 2^-133; one FMA makes it (q - 8) / 64 exactly.  64 s
// (11 bits) = hi + lo exactly with hi = bf16(64 s); (q - 8) / 64 * lo is exact
// (4 + 4 bits), and the last FMA adds the exact product with hi and rounds.
__device__ __forceinline__ uint4 dequant8_bf16(uint32_t w, uint32_t hi, uint32_t lo) {
  const uint32_t even = w & 0x0F0F0F0Fu, odd = (w >> 4) & 0x0F0F0F0Fu;
  uint32_t o[4];
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    // bytes: code 2b, 0, code 2b + 1, 0 (a selector's top bit replicates the
    // byte's sign, 0)
    uint32_t v;
    const uint32_t sel = b | ((8 + b) << 4) | ((4 + b) << 8) | ((12 + b) << 12);
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(v) : "r"(even), "r"(odd), "r"(sel));
    v = fma_bf16x2(v, 0x7F007F00u, 0xBE00BE00u);  // q 2^-133 * 2^127 - 8 / 64
    o[b] = fma_bf16x2(v, hi, mul_bf16x2(v, lo));
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}

// 32 codes of a row under one fp16 scale -> 16 TMEM columns of the thread's lane.
__device__ __forceinline__ void convert32(const uint4& c, uint32_t scale, uint32_t dst) {
  const float s = 64.0f * __half2float(__ushort_as_half((unsigned short)scale));
  const uint32_t hi = pack_bf16x2(s, s);
  const float rest = s - bf16_lo(hi);
  const uint32_t lo = pack_bf16x2(rest, rest);
  const uint4 a0 = dequant8_bf16(c.x, hi, lo), a1 = dequant8_bf16(c.y, hi, lo);
  const uint4 a2 = dequant8_bf16(c.z, hi, lo), a3 = dequant8_bf16(c.w, hi, lo);
  const uint32_t o[16] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w,
                          a2.x, a2.y, a2.z, a2.w, a3.x, a3.y, a3.z, a3.w};
  tmem_st16(dst, o);
}

// One arrival counting for `count` expected arrivals.
__device__ __forceinline__ void mbar_arrive_n(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// A conversion warp's waits, conversions and arrivals (ColsConvert).
struct ConvertOps {
  uint64_t *wfull, *wempty, *sempty, *afull;  // afull: the set's
  volatile int* abort_flag;
  const FusedArgs& a;  // 4-bit rings are powers of two
  uint32_t half, sw, ss, dst, x0, x[4];
  int lane, at;

  __device__ __forceinline__ bool slot(uint32_t w) const {
    return mbar_wait_warp(&wfull[w & (a.ring_w - 1)], (w & a.ring_w) != 0, abort_flag, a.wait_limit);
  }
  __device__ __forceinline__ bool stage(uint32_t st) const {
    return st < 2 || mbar_wait_warp(&sempty[(st - 2) & (a.ring_s - 1)], ((st - 2) & a.ring_s) != 0, abort_flag, a.wait_limit);
  }
  __device__ __forceinline__ void codes(uint32_t w, bool any) const {
    const uint32_t wi = w & (a.ring_w - 1);
    if (any) {
      tc_fence_after();
      // half a slot: 128 codes and four scales of the row
      const uint32_t src = sw + wi * kCSlot + at * 128 + ((half << 6) ^ x0);
      const uint2 sc = ld_shared_v2(ss + wi * kCScale + at * 16 + half * 8);
      const uint4 c0 = ld_shared_v4(src + x[0]), c1 = ld_shared_v4(src + x[1]);
      convert32(c0, sc.x & 0xFFFFu, dst);
      const uint4 c2 = ld_shared_v4(src + x[2]);
      convert32(c1, sc.x >> 16, dst + 16);
      const uint4 c3 = ld_shared_v4(src + x[3]);
      convert32(c2, sc.y & 0xFFFFu, dst + 32);
      convert32(c3, sc.y >> 16, dst + 48);
      tmem_st_wait();
      tc_fence_before();
    }
    __syncwarp();
    if (lane == 0) {
      mbar_arrive(afull);
      mbar_arrive_n(&wempty[wi], 2);  // the warp's rows of the slot are consumed, for two sets
    }
  }
  __device__ __forceinline__ void rows(uint32_t w, uint32_t j) const {
    tc_fence_after();
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const uint32_t src = sw + (w & (a.ring_w - 1)) * kCSlot + at * 128 + ((p << 6) ^ x0);
      const uint4 b0 = ld_shared_v4(src + x[0]), b1 = ld_shared_v4(src + x[1]);
      const uint4 b2 = ld_shared_v4(src + x[2]), b3 = ld_shared_v4(src + x[3]);
      const uint32_t o[16] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w,
                              b2.x, b2.y, b2.z, b2.w, b3.x, b3.y, b3.z, b3.w};
      tmem_st16(dst + j * 32 + 16 * p, o);
    }
    tmem_st_wait();
    tc_fence_before();
    __syncwarp();
    if (lane == 0 && j) mbar_arrive(afull);
  }
  __device__ __forceinline__ void none() const {
    if (lane == 0) mbar_arrive(afull);
  }
  __device__ __forceinline__ void pass(uint32_t w) const {
    if (lane == 0) mbar_arrive(&wempty[w & (a.ring_w - 1)]);
  }
};

__device__ __forceinline__ void st_shared_u16(uint32_t addr, uint32_t v) {
  asm volatile("{\n\t.reg .b16 h;\n\tcvt.u16.u32 h, %1;\n\tst.shared.b16 [%0], h;\n\t}" ::"r"(addr), "r"(v)
               : "memory");
}

__device__ __forceinline__ int ld_acquire_gpu(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release_gpu_add(int* p, int v) {
  asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ float silu_mul(float g, float u) {
  // approximate divide (2 ulp): far below the bf16 rounding of h; an infinite
  // e^-g (g < -88) gives 0, the limit of silu
  return __fdividef(g * u, 1.0f + __expf(-g));
}

// Group table of the launch (shared memory): the groups that have tiles, in
// order, the shared expert last.  A wave's (W: WaveParams) re-checks each slot (fail closed:
// a group whose slot does not hold the expected object and version gets no
// tiles, and CTA 0 records the lowest such expert's status).  Every thread
// calls it; returns the number of routed groups.
template <typename W>
__device__ __forceinline__ int cols_group_table(const FusedArgs& a, const W& w, bool record, int* s_mt,
                                                int* s_slot, int* s_rb, int* s_cnt, int* s_tmp) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  constexpr bool wave = std::is_same<W, WaveParams>::value;
  int n = a.num_groups;
  if constexpr (wave) n = w.n;
  int groups = 0, tiles = 0, kmin = 0x7fffffff;
  for (int i0 = 0; i0 < n; i0 += blockDim.x) {
    const int i = i0 + tid;
    int cnt = 0, slot = 0, rb = 0, code = 0, e = 0;
    if (i < n) {
      if constexpr (wave) {
        e = w.expert[i];
        cnt = a.counts[e];
        rb = a.offsets[e];
        slot = w.slot[i];
        if (cnt > 0) {
          if (slot < 0) {
            code = MSI_ERR_NOT_RESIDENT;
          } else {
            const unsigned long long obj = a.genwords[slot].obj;
            const unsigned long long gen = a.genwords[slot].gen;
            if (obj != obj_key(w.layer, e)) code = MSI_ERR_WRONG_OBJECT;
            else if (gen != w.expected[i]) code = MSI_ERR_STALE_GENERATION;
          }
        }
        if (code) cnt = 0;
      } else {
        const Group G = a.groups[i];
        cnt = G.ok ? G.row_count : 0;
        slot = G.slot;
        rb = G.row_begin;
      }
    }
    const int mt = (cnt + a.tile_tok - 1) / a.tile_tok;
    // block-wide exclusive positions: groups with tiles, and tiles
    const unsigned has = __ballot_sync(0xffffffffu, mt > 0);
    int incl = mt;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += o;
    }
    int key = code ? (e << 4) | code : 0x7fffffff;
    key = __reduce_min_sync(0xffffffffu, key);
    __syncthreads();  // the previous round's readers of s_tmp
    if (lane == 31) s_tmp[warp] = incl;
    if (lane == 0) {
      s_tmp[32 + warp] = __popc(has);
      s_tmp[64 + warp] = key;
    }
    __syncthreads();
    int gb = groups, tb = tiles;
    for (int q = 0; q < nw; ++q) {
      if (q < warp) {
        tb += s_tmp[q];
        gb += s_tmp[32 + q];
      }
      tiles += s_tmp[q];
      groups += s_tmp[32 + q];
      kmin = min(kmin, s_tmp[64 + q]);
    }
    if (mt > 0) {
      const int g = gb + __popc(has & ((1u << lane) - 1u));
      s_mt[g] = tb + incl - mt;
      s_slot[g] = slot;
      s_rb[g] = rb;
      s_cnt[g] = cnt;
    }
  }
  if (tid == 0) {
    s_mt[groups] = tiles;
    s_slot[groups] = a.sh_slot;  // the shared expert's, when there is one
    s_rb[groups] = 0;
    s_cnt[groups] = a.sh_rows;
    if (record && kmin != 0x7fffffff) atomicCAS(a.status, 0, kmin & 15);
  }
  return groups;
}

}  // namespace

// GATHER: x by TMA gathers (tiles of up to 64 tokens)
template <bool Q4, int STEPS, bool GATHER, typename W>
__global__ void __launch_bounds__(cols_threads(Q4), 1)
    fused_cols_kernel(const __grid_constant__ CUtensorMap tmW13, const __grid_constant__ CUtensorMap tmW2,
                      const __grid_constant__ CUtensorMap tmS13, const __grid_constant__ CUtensorMap tmS2,
                      const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmH,
                      const __grid_constant__ CUtensorMap tmHS, const __grid_constant__ FusedArgs a,
                      const __grid_constant__ W w) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  // stages: [bf16: steps x 16 KB of weights][steps x b_rows x 128 B of tokens]
  const int w_stage = Q4 ? 0 : STEPS * kCSlot;
  const int b_step = a.b_rows * 128;
  const int stage = w_stage + STEPS * b_step;
  uint8_t* sT = smem;
  uint8_t* sW = sT + a.ring_s * stage;   // 4-bit: [ring_w][128][128] codes
  uint8_t* sS = sW + a.ring_w * kCSlot;  // 4-bit: [ring_w][128][8] fp16 scales
  uint8_t* s_epi = sS + a.ring_w * kCScale;  // epilogue staging, 1 KB per warp
  uint64_t* sfull = reinterpret_cast<uint64_t*>(s_epi + 4096);  // [ring_s]
  uint64_t* sempty = sfull + kCRingMax;
  uint64_t* wfull = sempty + kCRingMax;   // 4-bit: [ring_w]
  uint64_t* wempty = wfull + kCRingMax;
  uint64_t* tfull = wempty + kCRingMax;   // [2]
  uint64_t* tempty = tfull + 2;           // [2]
  uint64_t* afull = tempty + 2;           // [4] 4-bit: a stage's steps in TMEM
  uint64_t* drain = afull + 4;
  uint64_t* never = drain + 1;  // no thread ever arrives here
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(never + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* s_mt = reinterpret_cast<int*>(tmem_slot + 2);  // [groups + 1]
  int* s_slot = s_mt + kCTable + 1;
  int* s_rb = s_slot + kCTable;
  int* s_cnt = s_rb + kCTable;
  int* s_tmp = s_cnt + kCTable;  // [96]

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < a.ring_s; ++s) {
      mbar_init(&sfull[s], kCTokWarps * (GATHER ? 1 : 32) + (Q4 ? 0 : 1));
      mbar_init(&sempty[s], 1);
    }
    for (int s = 0; s < a.ring_w; ++s) {
      mbar_init(&wfull[s], 33);  // the TMA and 32 lanes' scale copies
      mbar_init(&wempty[s], kCDqWarps);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], 4);
    }
    for (int s = 0; s < kCOperand; ++s) mbar_init(&afull[s], 4);
    mbar_init(drain, 1);
    mbar_init(never, 1);
    *abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 4) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  if (warp == 5 && lane == 0) {
    tma_prefetch(&tmW13);
    tma_prefetch(&tmW2);
    if (a.sh_rows > 0) {
      tma_prefetch(&tmS13);
      tma_prefetch(&tmS2);
    }
    tma_prefetch(&tmX);
    tma_prefetch(&tmH);
  }
  grid_wait();
  grid_release();
  // the previous wave's counters, zeroed for the next wave
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < a.n_ready_clear; r += gridDim.x * blockDim.x)
    a.ready_clear[r] = 0;
  const int ng = cols_group_table(a, w, blockIdx.x == 0, s_mt, s_slot, s_rb, s_cnt, s_tmp);
  const int g_sh = ng;  // the shared expert's group, when there is one
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const long long lim = a.wait_limit;
  ColsWalk walk;
  walk.init(s_mt, ng, (a.sh_rows + a.tile_tok - 1) / a.tile_tok, a.nt_up, a.nt_dn, gridDim.x, blockIdx.x, a.sched_w);

  if (warp == 5) {
    // ------------------------------------------------------------- weights
    if (!Q4) {
      if (lane == 0) {
        Ring r(a.ring_s);
        int issued = 0;
        bool ok = true;
        while (ok && walk.next()) {
          const ColsTile& t = walk.t;
          const bool sh = t.g == g_sh;
          const int kb_n = t.up ? a.kb_up : a.kb_dn;
          const int slot = s_slot[t.g];
          const CUtensorMap* map = sh ? (t.up ? &tmS13 : &tmS2) : (t.up ? &tmW13 : &tmW2);
          // first weight row: of the gate rows (the up rows follow I rows on), or of W2
          const int row = t.up ? slot * a.w13_rows_per_slot + t.n * 64
                               : slot * a.w2_rows_per_slot + a.w2_row_off + t.n * 128;
          for (int k0 = 0; k0 < kb_n; k0 += STEPS) {
            if (!mbar_wait(&sempty[r.i], r.ph ^ 1, abort_flag, lim)) { ok = false; break; }
            const int k1 = min(kb_n, k0 + STEPS);
            mbar_arrive_expect_tx(&sfull[r.i], (k1 - k0) * kCSlot);
            uint8_t* dst = sT + r.i * stage;
            for (int kb = k0; kb < k1; ++kb, dst += kCSlot) {
              if (!t.up) {
                tma_load_2d(dst, map, &sfull[r.i], kb * 64, row);
              } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                  tma_load_4d(dst + j * (kCSlot / 4), map, &sfull[r.i], kb * 64, 0, row / 16 + j, 0);
              }
            }
            r.step();
            ++issued;
          }
        }
        // on abort, the loads this thread armed land (bounded) before the
        // CTA's shared memory is released
        if (*abort_flag) {
          for (int d = 0; d < a.ring_s && d < issued; ++d) {
            const int j = issued - 1 - d;
            const long long t0 = clock64();
            while (!mbar_try_wait(&sfull[j % a.ring_s], (j / a.ring_s) & 1) && clock64() - t0 < kDrainCycles) {
            }
          }
        }
      }
    } else {
      // lane 0 issues the TMA loads; every lane copies four rows' scales of the
      // slot (cp.async, arriving on the slot's barrier as they land)
      Ring r(a.ring_w);
      int issued = 0;
      bool ok = true;
      while (ok && walk.next()) {
        const ColsTile& t = walk.t;
        const bool codes = t.g != g_sh;
        const int kb_n = t.up ? a.kb_up : a.kb_dn;
        const int slots = codes ? (kb_n + 3) / 4 : kb_n;  // 256 codes or 64 weights a slot
        const int slot = s_slot[t.g];
        const CUtensorMap* map = codes ? (t.up ? &tmW13 : &tmW2) : (t.up ? &tmS13 : &tmS2);
        const int row = t.up ? slot * (codes ? a.q13_rows_per_slot : a.w13_rows_per_slot) + t.n * 64
                             : (codes ? slot * a.q2_rows_per_slot + a.q2_row_off
                                      : slot * a.w2_rows_per_slot + a.w2_row_off) + t.n * 128;
        const uint8_t* sc[4];  // scales of the lane's four rows (slot rows lane + 32 i)
        const int sc_ld = t.up ? a.q13_scale_ld : a.q2_scale_ld;
        if (codes) {
          const uint8_t* base = a.q4_pool + (unsigned long long)slot * a.q4_extent +
                                (t.up ? a.q13_scale_off : a.q2_scale_off);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int rr = lane + 32 * i;
            sc[i] = base + (size_t)(t.up ? t.n * 64 + (rr & 63) + (rr >= 64 ? a.w13_up_off : 0) : t.n * 128 + rr) * sc_ld;
          }
        }
        for (int s = 0; s < slots; ++s) {
          if (!mbar_wait(&wempty[r.i], r.ph ^ 1, abort_flag, lim)) { ok = false; break; }
          if (lane == 0) {
            mbar_arrive_expect_tx(&wfull[r.i], kCSlot);
            uint8_t* dst = sW + r.i * kCSlot;
            const int k = codes ? s * 128 : s * 64;
            if (!t.up) {
              tma_load_2d(dst, map, &wfull[r.i], k, row);
            } else {
              tma_load_2d(dst, map, &wfull[r.i], k, row);
              tma_load_2d(dst + kCSlot / 2, map, &wfull[r.i], k, row + a.w13_up_off);
            }
          }
          if (codes) {
            uint8_t* dst = sS + r.i * kCScale + lane * 16;
            // the K's scales end inside the last slot when K is an odd
            // multiple of 128, and rows are then 8-byte aligned only
            const int left = sc_ld - s * 16;
            if (sc_ld % 16 == 0) {
#pragma unroll
              for (int i = 0; i < 4; ++i) cp_async16(dst + i * 512, sc[i] + s * 16, 16);
            } else {
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                cp_async8(dst + i * 512, sc[i] + s * 16);
                if (left >= 16) cp_async8(dst + i * 512 + 8, sc[i] + s * 16 + 8);
              }
            }
          }
          cp_async_arrive_noinc(&wfull[r.i]);
          r.step();
          ++issued;
        }
      }
      cp_async_wait<0>();
      if (*abort_flag && lane == 0) {
        for (int d = 0; d < a.ring_w && d < issued; ++d) {
          const int j = issued - 1 - d;
          const long long t0 = clock64();
          while (!mbar_try_wait(&wfull[j % a.ring_w], (j / a.ring_w) & 1) && clock64() - t0 < kDrainCycles) {
          }
        }
      }
    }
  } else if (warp == 4) {
    // ------------------------------------------------------------- MMA issuer
    // the whole warp walks and waits, so that the loop's state is uniform; one
    // lane issues
    Ring r(a.ring_s), ra(kCOperand);
    uint32_t acc = 0, aph = 0;
    const uint32_t desc_hi = (uint32_t)(sw128_desc(0) >> 32);
    const uint32_t s_lo = uniform((uint32_t)sw128_desc(smem_u32(sT)));
    const uint32_t tm = uniform(tmem_base);
    bool ok = true;
    while (ok && __any_sync(0xffffffffu, walk.next())) {
      const ColsTile& t = walk.t;
      const int kb_n = (int)uniform(t.up ? a.kb_up : a.kb_dn);
      const uint32_t cols = uniform(min(a.tile_tok, s_cnt[t.g] - t.m * a.tile_tok));
      const uint32_t idesc = idesc_bf16(128, (cols + 15) & ~15);
      ok = mbar_wait_warp(&tempty[acc], aph ^ 1, abort_flag, lim);
      if (!ok) break;
      const uint32_t d = tm + acc * 128;
      for (int k0 = 0; k0 < kb_n; k0 += STEPS) {
        ok = mbar_wait_warp(&sfull[r.i], r.ph, abort_flag, lim);
        if (!ok) break;
        // cp.async (generic proxy) wrote the tokens: before the tensor core's reads
        if (!GATHER) fence_proxy_async_smem();
        const uint32_t w_lo = s_lo + ((r.i * stage) >> 4);
        const uint32_t bl = w_lo + (w_stage >> 4);
        if (Q4) {
          // halves of two steps, as the conversion sets finish them (a stage
          // past the tile's K has its second half announced empty)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            ok = mbar_wait_warp(&afull[ra.i], ra.ph, abort_flag, lim);
            if (!ok) break;
            tc_fence_after();
            const uint32_t at = tm + kCOperandCol + ra.i * 64;
            if (elect_one()) {
              if (h == 0 || k0 + 2 < kb_n) {
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                  const uint32_t bj = bl + (2 * h + j) * (b_step >> 4);
#pragma unroll
                  for (int k = 0; k < 4; ++k)
                    umma_bf16_ts(d, at + 32 * j + 8 * k, desc64(bj + 2 * k, desc_hi), idesc, (k0 | h | j | k) != 0);
                }
              }
              if (h == 1) umma_commit(&sempty[r.i]);
            }
            __syncwarp();
            ra.step();
          }
          if (!ok) break;
        } else {
          tc_fence_after();
          if (elect_one()) {
#pragma unroll
            for (int j = 0; j < STEPS; ++j) {
              if (j < 2 || k0 + j < kb_n) {
                const uint32_t bj = bl + j * (b_step >> 4), wj = w_lo + j * (kCSlot >> 4);
#pragma unroll
                for (int k = 0; k < 4; ++k)
                  umma_bf16(d, desc64(wj + 2 * k, desc_hi), desc64(bj + 2 * k, desc_hi), idesc, (k0 | j | k) != 0);
              }
            }
            umma_commit(&sempty[r.i]);
          }
          __syncwarp();
        }
        r.step();
      }
      if (!ok) break;
      if (elect_one()) umma_commit(&tfull[acc]);
      __syncwarp();
      acc ^= 1;
      if (acc == 0) aph ^= 1;
    }
    // every MMA this warp issued has completed before TMEM is released
    __syncwarp();
    if (elect_one()) {
      umma_commit(drain);
      const long long t0 = clock64();
      while (!mbar_try_wait(drain, 0) && clock64() - t0 < kDrainCycles) {
      }
    }
  } else if (warp < 4) {
    // ------------------------------------------------------------- epilogue
    uint32_t jt = 0;
    const uint32_t stg = smem_u32(s_epi) + warp * 1024;
    if (a.stall && threadIdx.x == 0) mbar_wait(never, 0, abort_flag, lim);  // runs out: abort
    __syncwarp();
    while (walk.next()) {
      const ColsTile& t = walk.t;
      const bool sh = t.g == g_sh;
      const int row0 = t.m * a.tile_tok;
      const int rows = min(a.tile_tok, s_cnt[t.g] - row0);
      const uint32_t acc = jt & 1, aph = (jt >> 1) & 1;
      if (!mbar_wait_warp(&tfull[acc], aph, abort_flag, lim)) break;
      tc_fence_after();
      const uint32_t tb = tmem_base + ((uint32_t)(warp * 32) << 16) + acc * 128;
      const size_t orow = (size_t)(sh ? row0 : s_rb[t.g] + row0);
      // sixteen tokens at a time through the warp's staging buffer, [token][its
      // weight rows' bf16], so that a store fills 32 or 64 contiguous bytes a
      // token with one 16-byte store a lane (a 2- or 4-byte store per token and
      // lane took the epilogue warps 92 % of the time at 4,096 tokens)
      if (t.up) {
        const int half = lane >> 4;  // 0: the lane's row is a gate row, 1: an up row
        const uint32_t put = stg + half * 32 + (lane & 15) * 2;
        __nv_bfloat16* out = (sh ? a.hs : a.h) + orow * a.h_ld + t.n * 64 + warp * 16 + (lane & 1) * 8;
#pragma unroll 1
        for (int c = 0; c < rows; c += 16) {
          uint32_t v[16];
          tmem_ld16(tb + c, v);
          tmem_ld_wait(v);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            // gate lanes take the even token of a pair, up lanes the odd one
            const uint32_t o = __shfl_xor_sync(0xffffffffu, half ? v[2 * i] : v[2 * i + 1], 16);
            const float g = __uint_as_float(half ? o : v[2 * i]);
            const float u = __uint_as_float(half ? v[2 * i + 1] : o);
            st_shared_u16(put + i * 64, pack_bf16x2(silu_mul(g, u), 0.f));
          }
          __syncwarp();
          const int tok = c + (lane >> 1);
          const uint4 q = ld_shared_v4(stg + lane * 16);
          if (tok < rows) *reinterpret_cast<uint4*>(out + (size_t)tok * a.h_ld) = q;
          __syncwarp();
        }
        // publish the warp's part of the tile: its h stores, then one release
        // add on the token tile's counter
        __threadfence();
        __syncwarp();
        if (lane == 0) red_release_gpu_add(&a.ready[s_mt[t.g] + t.m], 1);
      } else {
        const uint32_t put = stg + lane * 2;
        __nv_bfloat16* out = (sh ? a.ys : a.y) + orow * a.y_ld + t.n * 128 + warp * 32 + (lane & 3) * 8;
#pragma unroll 1
        for (int c = 0; c < rows; c += 16) {
          uint32_t v[16];
          tmem_ld16(tb + c, v);
          tmem_ld_wait(v);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const uint32_t p = pack_bf16x2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
            st_shared_u16(put + i * 128, p);
            st_shared_u16(put + i * 128 + 64, p >> 16);
          }
          __syncwarp();
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const int tok = c + 8 * j + (lane >> 2);
            const uint4 q = ld_shared_v4(stg + j * 512 + lane * 16);
            if (tok < rows) *reinterpret_cast<uint4*>(out + (size_t)tok * a.y_ld) = q;
          }
          __syncwarp();
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tempty[acc]);
      ++jt;
    }
  } else if (warp < 6 + kCTokWarps) {
    // ------------------------------------------------------------- token rows
    const int tw = warp - 6;
    const int gt = threadIdx.x - 6 * 32;  // copies: 16-byte chunk gt % 8 of rows gt / 8 + 16 i
    const int chunk = gt & 7, r0 = gt >> 3;
    constexpr int kRows = GATHER ? 1 : 8;
    constexpr int kWarpArrivals = GATHER ? 1 : 32;
    Ring r(a.ring_s);
    int issued = 0;  // stages
    bool ok = true;
    // an up tile's tokens, loaded one tile ahead: of row 4 tw + 16 (lane / 4) +
    // lane % 4 (gather; past the tile its last row's), or of rows r0 + 16 i
    auto tile_rows = [&](const ColsTile& t, int (&tok)[kRows]) {
      if (!t.up) return;
      const int row0 = t.m * a.tile_tok;
      const int rows = min(a.tile_tok, s_cnt[t.g] - row0);
      const int* perm = a.perm + s_rb[t.g] + row0;
      if (GATHER) {
        const int rr = min(4 * tw + 16 * (lane >> 2) + (lane & 3), rows - 1);
        tok[0] = t.g == g_sh ? row0 + rr : perm[rr];
      } else {
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
          if (16 * i >= rows) break;
          const int rr = r0 + 16 * i;
          tok[i] = t.g == g_sh ? row0 + rr : rr < rows ? perm[rr] : 0;
        }
      }
    };
    int tok[kRows], tok_next[kRows];
    bool more = walk.next();
    if (more) tile_rows(walk.t, tok_next);
    while (more && ok) {
      const ColsTile t = walk.t;
      const bool sh = t.g == g_sh;
      const int rows = min(a.tile_tok, s_cnt[t.g] - t.m * a.tile_tok);
      const int kb_n = t.up ? a.kb_up : a.kb_dn;
      const int n_it = (rows + 15) >> 4;
#pragma unroll
      for (int i = 0; i < kRows; ++i) {
        if (i >= n_it) break;
        tok[i] = tok_next[i];
      }
      more = walk.next();
      if (more) tile_rows(walk.t, tok_next);
      if (!t.up) {
        // every up tile of this token tile has published its h columns
        if (lane == 0) {
          const int* rdy = a.ready + s_mt[t.g] + t.m;
          const long long t0 = clock64();
          while (ld_acquire_gpu(rdy) < 4 * a.nt_up) {
            if (*abort_flag) { ok = false; break; }
            if (clock64() - t0 > lim) {
              *abort_flag = 1;
              ok = false;
              break;
            }
          }
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
        __syncwarp();
        if (!ok) break;
        fence_proxy_async_global();
        // warp j loads the stage's step j in boxes of 16 rows (the last one's
        // rows past the tile's are another group's or the tensor's zero fill:
        // for columns that no output reads)
        const CUtensorMap* map = sh ? &tmHS : &tmH;
        const int row = (sh ? 0 : s_rb[t.g]) + t.m * a.tile_tok;
        for (int k0 = 0; k0 < kb_n; k0 += STEPS) {
          if (!mbar_wait_warp(&sempty[r.i], r.ph ^ 1, abort_flag, lim)) { ok = false; break; }
          if (elect_one()) {
            if (tw < STEPS && k0 + tw < kb_n) {
              mbar_arrive_expect_tx(&sfull[r.i], n_it * 2048);
              if (kWarpArrivals > 1) mbar_arrive_n(&sfull[r.i], kWarpArrivals - 1);
              uint8_t* dst = sT + w_stage + r.i * stage + tw * b_step;
              for (int i = 0; i < n_it; ++i)
                tma_load_2d(dst + i * 2048, map, &sfull[r.i], (k0 + tw) * kBK, row + 16 * i);
            } else {
              mbar_arrive_n(&sfull[r.i], kWarpArrivals);
            }
          }
          __syncwarp();
          r.step();
          ++issued;
        }
      } else if (GATHER) {
        // quads tw, tw + 4, ... of the tile's rows, one a lane
        const int nq = ((rows + 3) / 4 - tw + 3) / 4;
        const int q = 4 * (lane & 7);
        const int i0 = __shfl_sync(0xffffffffu, tok[0], q), i1 = __shfl_sync(0xffffffffu, tok[0], q + 1);
        const int i2 = __shfl_sync(0xffffffffu, tok[0], q + 2), i3 = __shfl_sync(0xffffffffu, tok[0], q + 3);
        const uint32_t dst0 = smem_u32(sT) + w_stage + tw * 512 + lane * 2048, bar0 = smem_u32(sfull);
        for (int k0 = 0; k0 < kb_n; k0 += STEPS) {
          if (!mbar_wait_warp(&sempty[r.i], r.ph ^ 1, abort_flag, lim)) { ok = false; break; }
          const int ks = min(STEPS, kb_n - k0);
          if (elect_one()) {
            if (nq > 0) mbar_arrive_expect_tx(&sfull[r.i], ks * nq * 512);
            else mbar_arrive(&sfull[r.i]);
          }
          __syncwarp();
          if (lane < nq) {
            uint32_t dst = dst0 + r.i * stage;
            for (int st = 0; st < ks; ++st, dst += b_step)
              tma_gather4(dst, &tmX, bar0 + r.i * 8, (k0 + st) * kBK, i0, i1, i2, i3);
          }
          __syncwarp();
          r.step();
          ++issued;
        }
      } else {
        const __nv_bfloat16* src[kRows];
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
          if (i >= n_it) break;
          src[i] = r0 + 16 * i < rows ? a.x + (size_t)tok[i] * a.x_ld + chunk * 8 : a.x;
        }
        const uint32_t dst0 = smem_u32(sT) + w_stage + r0 * 128 + ((chunk ^ (r0 & 7)) << 4);
        for (int k0 = 0; k0 < kb_n; k0 += STEPS) {
          if (!mbar_wait_warp(&sempty[r.i], r.ph ^ 1, abort_flag, lim)) { ok = false; break; }
          const uint32_t dst = dst0 + r.i * stage;
#pragma unroll
          for (int i = 0; i < kRows; ++i) {
            if (i >= n_it) break;
            const uint32_t bytes = r0 + 16 * i < rows ? 16u : 0u;
            cp_async16_at(dst + i * 2048, src[i], bytes);
            cp_async16_at(dst + b_step + i * 2048, src[i] + kBK, bytes);
            if (STEPS == 4 && k0 + 2 < kb_n) {
              cp_async16_at(dst + 2 * b_step + i * 2048, src[i] + 2 * kBK, bytes);
              cp_async16_at(dst + 3 * b_step + i * 2048, src[i] + 3 * kBK, bytes);
            }
            src[i] += STEPS * kBK;
          }
          cp_async_arrive_noinc(&sfull[r.i]);  // arrives when this thread's copies land
          r.step();
          ++issued;
        }
      }
    }
    if (!GATHER) cp_async_wait<0>();
    // on abort, the loads this warp issued land (bounded), as above
    if (*abort_flag && lane == 0) {
      for (int d = 0; d < a.ring_s && d < issued; ++d) {
        const int j = issued - 1 - d;
        const long long t0 = clock64();
        while (!mbar_try_wait(&sfull[j % a.ring_s], (j / a.ring_s) & 1) && clock64() - t0 < kDrainCycles) {
        }
      }
    }
  } else if (Q4) {
    // ------------------------------------------------------------- conversion
    const int q = warp & 3;                   // TMEM lane quarter
    const uint32_t set = (warp - kCDqWarp0) >> 2;
    ColsConvert conv(set);
    ConvertOps op{wfull, wempty, sempty, afull + set, abort_flag, a};
    op.lane = lane;
    op.half = conv.half;
    op.sw = smem_u32(sW);
    op.ss = smem_u32(sS);
    op.dst = tmem_base + ((uint32_t)(q * 32) << 16) + kCOperandCol + set * 64;
    // the thread's row in a slot: down tiles in order, up tiles 64 gate rows,
    // then 64 up rows; 16-byte chunk c of row r lies at chunk c ^ (r & 7)
    const int at_dn = q * 32 + lane, at_up = (lane >> 4) * 64 + q * 16 + (lane & 15);
    op.x0 = (lane & 4) << 4;
#pragma unroll
    for (int c = 0; c < 4; ++c) op.x[c] = ((uint32_t)c ^ (lane & 3u)) << 4;
    while (walk.next()) {
      const ColsTile& t = walk.t;
      op.at = t.up ? at_up : at_dn;
      if (!conv.tile(t.g != g_sh, t.up ? a.kb_up : a.kb_dn, op)) break;
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 4) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
  if (threadIdx.x == 0 && *abort_flag) atomicCAS(a.status, 0, (int)MSI_ERR_TIMEOUT);
}

namespace {

constexpr int kColsFixed = 1024 + 4096 + (4 * kCRingMax + 4 + 4 + 2) * 8 + 8 + (4 * kCTable + 1 + 96) * 4;
constexpr int kColsSmem = 227 * 1024;

template <bool Q4, int STEPS, bool GATHER, typename W>
cudaError_t launch_cols(const CUtensorMap& tmW13, const CUtensorMap& tmW2, const CUtensorMap& tmS13,
                        const CUtensorMap& tmS2, const CUtensorMap& tmX, const CUtensorMap& tmH,
                        const CUtensorMap& tmHS, const FusedArgs& a, const W& w, int grid, bool after,
                        cudaStream_t s) {
  static std::atomic<unsigned long long> attr_done{0};
  cudaError_t e = smem_attr_once(fused_cols_kernel<Q4, STEPS, GATHER, W>, kColsSmem, attr_done);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeCooperative;  // every CTA resident: see above
  attr[0].val.cooperative = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3(cols_threads(Q4), 1, 1);
  cfg.dynamicSmemBytes = kColsFixed + a.ring_s * STEPS * ((Q4 ? 0 : kCSlot) + a.b_rows * 128) + a.ring_w * (kCSlot + kCScale);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = after ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, fused_cols_kernel<Q4, STEPS, GATHER, W>, tmW13, tmW2, tmS13, tmS2, tmX, tmH, tmHS, a, w);
}

}  // namespace

// Tokens per tile and stages of a launch of `rows` rows over `groups` experts
// of a call of T tokens.  A tile of as few tokens as most experts have leaves
// room for more stages of more K each; a group with more rows takes several
// tiles (and converts or reads its weights for each).  4-bit: at least as many
// stages as the TMEM ring holds, the rest of shared memory to codes in flight;
// from 24 rows a group on 128-token tiles (the call at 1,600 tokens, 31 rows a
// group, 406 us against 426 with 64; at 1,200 388 both).
int cols_tile_tokens(long long rows, int groups) {
  return rows <= 10LL * groups ? 32 : rows <= 24LL * groups ? 64 : 128;
}

void cols_rings(FusedArgs& a, bool q4, int T) {
  a.b_rows = T >= a.tile_tok ? a.tile_tok : (T + 15) / 16 * 16;
  const int room = kColsSmem - kColsFixed;
  if (q4) {
    a.steps = 4;
    const int tok = a.steps * a.b_rows * 128;
    a.ring_s = a.b_rows > 32 ? 2 : 4;
    a.ring_w = room - a.ring_s * tok >= 8 * (kCSlot + kCScale) ? 8 : 4;
  } else {
    a.steps = a.b_rows > 16 ? 2 : 4;
    const int fit = room / (a.steps * (kCSlot + a.b_rows * 128));
    a.ring_s = fit < kCRingMax ? fit : kCRingMax;
    a.ring_w = 0;
  }
}

cudaError_t launch_fused_cols(bool q4, const CUtensorMap& tmW13, const CUtensorMap& tmW2, const CUtensorMap& tmS13,
                              const CUtensorMap& tmS2, const CUtensorMap& tmX, const CUtensorMap& tmH,
                              const CUtensorMap& tmHS, const FusedArgs& a, const WaveParams& w, int grid, bool after,
                              cudaStream_t s) {
  if (grid < 1) return cudaSuccess;
  const auto go = [&](auto launch, const auto& wave) {
    return launch(tmW13, tmW2, tmS13, tmS2, tmX, tmH, tmHS, a, wave, grid, after, s);
  };
  if (!q4)
    return a.steps == 4 ? go(launch_cols<false, 4, true, NoWave>, NoWave{})
                        : go(launch_cols<false, 2, true, NoWave>, NoWave{});
  if (a.tile_tok > 64)
    return a.wave ? go(launch_cols<true, 4, false, WaveParams>, w) : go(launch_cols<true, 4, false, NoWave>, NoWave{});
  return a.wave ? go(launch_cols<true, 4, true, WaveParams>, w) : go(launch_cols<true, 4, true, NoWave>, NoWave{});
}

}  // namespace msi
