// Chunked prefill against the paged FP8 cache on the 5th-generation tensor cores: Eq. 1 with the causal K_{<=t}, Eq. 6
// dequantisation on load, Eq. 7-8 grouped-query sharing, Eq. 9 valid blocks only, Eq. 10 max-subtracted softmax, for runs
// of several query tokens per sequence.  head_dim 64 and 128.
//
// A CTA owns one (sequence, kv head) and two tiles of consecutive query tokens (or one, where all CTAs start at once).  The 128 rows of a tile are its (query
// token, query head of the group) pairs, so the K/V stream of the kv head is fetched, and V widened, once for all G heads
// and both tiles (Algorithm 2).  Per tile and 128 keys (eight cache blocks):
//     S [128 rows x 128 keys] = Q [128 x D] . Ktile^T       head_dim 128: kind::f8f6f4, the cache codes as they are, Q as
//                                                           two E4M3 terms of the bf16 query; head_dim 64: kind::f16, Q and
//                                                           K in f16 (both exact)
//     O [128 rows x D]       += P [128 x 128 keys] . Vtile  kind::f16: P rounded once to f16 and read from tensor memory, V
//                                                           codes widened to f16 (exact) in shared memory
// with fp32 accumulators in tensor memory.  The K scale of a block multiplies the logits of its 16 keys, the V scale goes
// into the exponent of the probabilities.
//
// What bounds it: per tile of 128 x 128 the exponential units need 1,024 cycles of an SM (16 a cycle) and the tensor core
// 1,024 (head_dim 64: 512).  Both run all the time only if neither waits for the other: a tile is multiplied 64 keys (a
// half) at a time, the logits two halves ahead of the softmax (one ahead, waiting for registers to take them: 447 us against
// 439), and two tiles share the SM.
// Softmax of a tile: four warps, one row per thread, the row's 64 logits of the half in registers, read once.  It keeps a
// reference maximum per row that may lag the true one by up to 2^11 (and a V scale reference that a scale may exceed by up
// to 2^4), so the accumulator in tensor memory is rescaled rarely; f16 probabilities have room for that factor.
//
// Tensor memory (512 columns): logits of tile x in two buffers of 64 columns from 128 x, the half's probabilities, two f16
// to a column, in the same place once the logits are in registers; its accumulator from 256 + D x.
//
// Warp roles (512 threads):
//   warps 0-3, 4-7   softmax of tile 0, of tile 1
//   warps 8-11       widen V (head_dim 64: and K) tiles into f16 operands
//   warps 12, 13     issue the matrix instructions of tile 0, of tile 1
//   warp 14          copies: gather requests over the tensor map of the cache
//   warp 15          what the softmax needs of a tile's block scales, worked out once for all rows
//
// Measured: 8 sequences of 4096 cached and 512 new tokens, 40 query heads over 8 kv heads, head_dim 128: 385 us (one tile a CTA,
// its key tiles taken in turns by two groups of eight warps: 690; the two tiles' exponentials side by side and one fp32
// operation an instruction: 412); prompts of 900..2900 tokens, 32 heads over 8, head_dim 64: 178 us (on mma.sync 495; 188).  A
// half takes about 1,700 cycles for both tiles: a softmax warp waits 300 for logits, loads them in 140, has their maximum in
// 240 more, and is 740 at the exponentials, 512 of which they need; shared memory is busy 1,600 cycles of it at head_dim 128
// (the products of Q, 64 keys at a time, read 6 KB each).  Half the exponentials left out took 12 % off, half the products of Q
// 4 %; four softmax warps a scheduler, two threads to a row, took 453 us against 439; a CTA's start and end take 15,000
// cycles (head_dim 64: 10,000).
// Every wait is bounded; a wait that runs out is reported in the status word and all roles leave through the common exit,
// which frees the tensor memory.
#include "coopt_umma.cuh"

namespace coopt {

namespace {

constexpr int kRows = 128;
constexpr int kThreads = 512;
constexpr int kWidenWarp = 8, kMmaWarp = 12, kCopyWarp = 14;      // warp 15: scales
constexpr int kTileBlocks = 8;
constexpr int kTileKeys = kTileBlocks * kBlockSize;        // 128: what is copied and widened at a time
constexpr int kHalf = kTileKeys / 2;                       // 64: what is multiplied at a time
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kMaxLag = 11.0f;                           // a row's reference may lag its maximum by this much (base-2 logarithm units)
constexpr float kScaleLag = 16.0f;                         // a V scale may exceed the reference scale by this factor

struct PrefillParams {
  const __nv_bfloat16* q;
  __nv_bfloat16* out;
  const int* cu_q_lens;
  const int* block_table;
  const int* context_lens;
  int max_blocks_per_seq;
  int batch, num_q_heads, num_kv_heads, group;
  int num_blocks;
  int tile_queries;        // query tokens per tile = 128 / group
  int tiles;               // of a CTA: 2, or 1
  int causal;
  int by_length;           // more CTAs than the device holds at a time: the long ones first
  float sm_scale_log2;
  int* status;
};

template <int D>
struct Cfg {
  static constexpr bool kWideK = D == 64;                         // K is widened to f16 too
  static constexpr int kPart = kBlockSize * D;                    // K (or V) codes of one granule
  static constexpr int kGran = granule_bytes(D, true);
  static constexpr int kCodes = kTileBlocks * kPart;              // K (or V) codes of a tile
  static constexpr int kKSlot = kCodes + kTileBlocks * kFp8Header;   // K parts, then the eight headers
  static constexpr int kKSlots = D == 128 ? 3 : 2, kVSlots = 2, kWide = 2, kScaleSlots = 4;
  static constexpr int kOperand = 128 * D * 2;                    // Q of a tile (two terms of codes, or f16); V^T, or K, of a tile in f16
  static constexpr int kKOff = 0;
  static constexpr int kVOff = kKOff + kKSlots * kKSlot;
  static constexpr int kQOff = kVOff + kVSlots * kCodes;
  static constexpr int kV16Off = kQOff + 2 * kOperand;
  static constexpr int kK16Off = kV16Off + kWide * kOperand;
  static constexpr int kScaleOff = kK16Off + (kWideK ? kWide * kOperand : 0);   // [slot][32]: K scales, log2 of V scale ratios, their inverses, factor, reference
  static constexpr int kBarOff = kScaleOff + kScaleSlots * 128;
  static constexpr int kNumBars = 2 * kKSlots + 2 * kVSlots + 4 * kWide + kScaleSlots + 21;
  static constexpr int kMiscOff = kBarOff + kNumBars * 8;
  static constexpr int kSmemBytes = kMiscOff + 64;
  static_assert(kKSlot % 128 == 0 && kVOff % 128 == 0 && kQOff % 128 == 0 && kSmemBytes <= 232448, "shared memory of one CTA");
};

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
                 "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Four codes -> four f16 (exact).  Two cycles of a scheduler per conversion of two codes; integer instructions for the same
// (shift, mask, sign) take 14 cycles per four codes.
template <bool kE5m2>
__device__ __forceinline__ uint2 widen4(uint32_t w) {
  if (kE5m2) return make_uint2(e5m2x2_to_f16x2_lo(w), e5m2x2_to_f16x2_hi(w));
  return make_uint2(e4m3x2_to_f16x2_lo(w), e4m3x2_to_f16x2_hi(w));
}
// Two fp32 operations in one instruction.
__device__ __forceinline__ uint64_t f32_pair(float a, float b) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ float2 f32_both(uint64_t a) {
  float2 d;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(a));
  return d;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// A wait by all lanes of a warp, and an arrival by one of them (behind the others).
__device__ __forceinline__ bool wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  return __all_sync(0xffffffffu, wait_bar(bar, parity, abort_flag));
}
__device__ __forceinline__ void arrive_one(uint64_t* bar) {
  asm volatile("{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n @q mbarrier.arrive.shared::cta.b64 _, [%0];\n}" ::"r"(smem_u32(bar)) : "memory");
}

// kTurns: the two tiles of a CTA take turns at the exponentials.  A launch with one tile a CTA has a kernel without that code, which
// nothing waits in there but which costs all the same (256 new tokens behind 2 x 8192, G = 8, 115.4 / 113.2 us; 24 sequences of
// 335..671 tokens, one head, 23.8 / 23.4).
template <int D, bool kE5m2, bool kTurns>
__global__ void __launch_bounds__(kThreads, 1) paged_prefill_kernel(const PrefillParams p, const __grid_constant__ CUtensorMap map_part,
                                                                    const __grid_constant__ CUtensorMap map_hdr) {
  using C = Cfg<D>;
  extern __shared__ __align__(128) uint8_t smem[];
  float* scales = reinterpret_cast<float*>(smem + C::kScaleOff);
  uint64_t* bar_kfull = reinterpret_cast<uint64_t*>(smem + C::kBarOff);   // K parts and headers of a tile have landed
  uint64_t* bar_kfree = bar_kfull + C::kKSlots;         // .. are of no more use: to the scale warp, and to both tiles' products (or the widening warps)
  uint64_t* bar_vfull = bar_kfree + C::kKSlots;         // V parts of a tile have landed
  uint64_t* bar_vfree = bar_vfull + C::kVSlots;         // .. have been widened
  uint64_t* bar_v16full = bar_vfree + C::kVSlots;       // V operand ready
  uint64_t* bar_v16free = bar_v16full + C::kWide;       // .. both tiles' products with it are done
  uint64_t* bar_k16full = bar_v16free + C::kWide;       // the same of K
  uint64_t* bar_k16free = bar_k16full + C::kWide;
  uint64_t* bar_scale = bar_k16free + C::kWide;         // the softmax's share of a tile's scales is ready
  uint64_t* bar_sfull = bar_scale + C::kScaleSlots;     // [tile][buffer] logits of a half are in tensor memory (and the tile's scales ready)
  uint64_t* bar_pfull = bar_sfull + 4;                  // [tile][buffer] its probabilities are, in their place
  uint64_t* bar_pv = bar_pfull + 4;                     // [tile] its product with V is done
  uint64_t* bar_out = bar_pv + 2;                       // [tile] .. and it was the tile's last
  uint64_t* bar_q = bar_out + 2;                        // the query operands are in shared memory
  uint64_t* bar_turn = bar_q + 1;                       // [tile][scheduler] the exponentials of a half are done
  int* misc = reinterpret_cast<int*>(smem + C::kMiscOff);   // [0] sequence, [1] first query, [2] abort flag, [3] tensor memory, [4] first row, [5] rows, [6] context of the sequence, [7] kv head
  volatile int* abort_flag = misc + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(misc + 3);

  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;      // (the warp in a uniform register)
  const int G = p.group, Hq = p.num_q_heads, Hkv = p.num_kv_heads;
  const int TQ = p.tile_queries;

  if (tid == 0) {
    *abort_flag = 0;
    for (int i = 0; i < C::kKSlots; ++i) { mbar_init(&bar_kfull[i], 1); mbar_init(&bar_kfree[i], C::kWideK ? 5 : 3); }
    for (int i = 0; i < C::kVSlots; ++i) { mbar_init(&bar_vfull[i], 1); mbar_init(&bar_vfree[i], 4); }
    for (int i = 0; i < C::kWide; ++i) {
      mbar_init(&bar_v16full[i], 4); mbar_init(&bar_v16free[i], 2);
      mbar_init(&bar_k16full[i], 4); mbar_init(&bar_k16free[i], 2);
    }
    for (int i = 0; i < C::kScaleSlots; ++i) mbar_init(&bar_scale[i], 1);
    mbar_init(bar_q, 8);
    for (int i = 0; i < 8; ++i) mbar_init(&bar_turn[i], 1);
    for (int i = 0; i < 4; ++i) { mbar_init(&bar_sfull[i], 2); mbar_init(&bar_pfull[i], 4); }
    for (int i = 0; i < 2; ++i) { mbar_init(&bar_pv[i], 1); mbar_init(&bar_out[i], 1); }
    mbar_fence_init();
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == kCopyWarp * 32) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_part) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_hdr) : "memory");
  }
  wait_previous_kernel();

  // softmax groups: this thread's row r of tile x
  const int x = warp >> 2, r = tid & (kRows - 1), qi = r / G, qh = r - qi * G;
  // ---- which (sequence, kv head, pair of query tiles) is this CTA's --------------------------------------------------------
  // Pairs with many keys to go through come first, over all sequences, so that the last CTAs to start are short ones.  How
  // many is a pair's level (in pairs of queries: what fits into the tokens up to it), and levels are taken an eighth of the
  // highest at a time: within that, the pairs of a (sequence, kv head) are neighbours and read its cache from L2 together.
  // (Sequence after sequence, prompts of 900..2900 tokens took 204 us, 24 sequences of 105..3158 tokens 115; in this order
  // 187 and 94; 8 sequences of 4096 + 512 tokens take 427 and 431 us, 443 level by level.)
  if (warp == 0) {
    constexpr int kPer = 4, kBands = 8;
    int left = blockIdx.x, found = -1, g = 0, q0 = 0, first = 0, count = 0, ctx = 0;
    const int W = p.tiles * TQ;
    auto sequence = [&](int b, int& from, int& n, int& c) {
      from = b < p.batch ? p.cu_q_lens[b] : 0;
      n = b < p.batch ? max(0, p.cu_q_lens[b + 1] - from) : 0;
      c = b < p.batch ? max(0, min(p.context_lens[b], p.max_blocks_per_seq * kBlockSize)) : 0;
    };
    // this CTA among those of 32 sequences, of which lane l's has the pairs [last - m + 1, last]
    auto look = [&](int b0, int m, int last, int from, int n, int c) {
      int upto = m * Hkv;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, upto, o);
        if (lane >= o) upto += t;
      }
      const unsigned in = __ballot_sync(0xffffffffu, upto > left);
      if (in == 0) { left -= __shfl_sync(0xffffffffu, upto, 31); return; }
      const int l = __ffs(in) - 1;
      m = __shfl_sync(0xffffffffu, m, l);
      left -= __shfl_sync(0xffffffffu, upto, l) - m * Hkv;
      found = b0 + l;
      g = left / m;
      q0 = (__shfl_sync(0xffffffffu, last, l) - left % m) * W;
      first = __shfl_sync(0xffffffffu, from, l);
      count = __shfl_sync(0xffffffffu, n, l);
      ctx = __shfl_sync(0xffffffffu, c, l);
    };
    if (p.by_length && p.batch <= 32 * kPer) {
      int from[kPer], n[kPer], c[kPer], pairs[kPer], end[kPer], top = 0;
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        sequence(32 * i + lane, from[i], n[i], c[i]);
        pairs[i] = (n[i] + W - 1) / W;
        end[i] = max(0, c[i] - n[i]) / W + pairs[i];
        top = max(top, end[i]);
      }
      const int width = max(1, (__reduce_max_sync(0xffffffffu, top) + kBands - 1) / kBands);
      auto above = [&](int i, int v) { return max(0, min(pairs[i], end[i] - v * width)); };      // pairs of band v and higher ones
      int band = kBands - 1;
#pragma unroll 1
      for (; band >= 0; --band) {
        int k = 0;
#pragma unroll
        for (int i = 0; i < kPer; ++i) k += above(i, band);
        if (static_cast<int>(__reduce_add_sync(0xffffffffu, k)) * Hkv > left) break;
      }
      if (band >= 0) {
        int k = 0;
#pragma unroll
        for (int i = 0; i < kPer; ++i) k += above(i, band + 1);
        left -= static_cast<int>(__reduce_add_sync(0xffffffffu, k)) * Hkv;
#pragma unroll
        for (int i = 0; i < kPer; ++i)
          if (found < 0) look(32 * i, above(i, band) - above(i, band + 1), pairs[i] - 1 - above(i, band + 1), from[i], n[i], c[i]);
      }
    } else {
      // all CTAs start at once, or so many sequences that each is short against the whole: one after the other, each from its end
      for (int b0 = 0; b0 < p.batch && found < 0; b0 += 32) {
        int from, n, c;
        sequence(b0 + lane, from, n, c);
        const int pairs = (n + W - 1) / W;
        look(b0, pairs, pairs - 1, from, n, c);
      }
    }
    if (lane == 0) { misc[0] = found; misc[1] = q0; misc[4] = first; misc[5] = count; misc[6] = ctx; misc[7] = g; }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int b = misc[0], q0 = misc[1], row_base = misc[4], n_new = misc[5], L = misc[6], g = misc[7];
  // keys that any row of tile x may see (Eq. 1: K_{<=t}), and tiles of keys
  auto tile_queries = [&](int x) { return x < p.tiles ? max(0, min(TQ, n_new - q0 - x * TQ)) : 0; };
  auto tile_keys = [&](int x) {
    const int nq = tile_queries(x);
    return nq == 0 ? 0 : p.causal ? max(0, min(L, L - n_new + q0 + x * TQ + nq)) : L;
  };
  const int kv_end = max(tile_keys(0), tile_keys(1));
  const int n_blocks = (kv_end + kBlockSize - 1) / kBlockSize, n_tiles = (kv_end + kTileKeys - 1) / kTileKeys;

  const bool live = x < 2 && qi < tile_queries(x);
  const size_t grow = static_cast<size_t>(row_base + q0 + x * TQ + (live ? qi : 0)) * Hq + g * G + (live ? qh : 0);
  uint32_t pend_mask = 0, pend_par = 0;                 // copy lane: the latest phase expected of every slot it has filled

  if (n_tiles == 0) {
    // no such tile, or nothing visible: all-zero rows
    if (live)
      for (int d = 0; d < D; d += 8) *reinterpret_cast<uint4*>(p.out + grow * D + d) = make_uint4(0u, 0u, 0u, 0u);
  } else if (warp < 8) {
    // ================= softmax: one row per thread ===================================================================
    asm volatile("setmaxnreg.inc.sync.aligned.u32 168;");
    const uint32_t lane_base = static_cast<uint32_t>(warp & 3) * 32u << 16;
    const uint32_t s_cols = tmem + 2 * kHalf * x + lane_base, o_cols = tmem + 4 * kHalf + D * x + lane_base;
    // ---- the query operand of the warp's 32 rows, eight at a time: a lane has every fourth 16 bytes of one of them.  The bf16
    // rows come into the operand's own place first.  (Loops that are not unrolled: code that a CTA runs once is bound by the
    // fetch of its instructions, about four cycles each.  A row per lane and all of it unrolled: 12,000 cycles, head_dim 64
    // 5,500.)
    const int row_off = live ? qi * Hq + qh : -1;      // from the tile's first row
    const size_t tile_row = static_cast<size_t>(row_base + q0 + x * TQ) * Hq + g * G;
    float qscale = 0.0f;       // logits of this row = tensor-memory value * qscale * K scale of the block
    {
      constexpr int kOctet = (C::kWideK ? 16 : 8) * D;    // eight rows of the operand (head_dim 128: of one term)
      const int row = lane & 7, at = lane >> 3;
      uint8_t* operand = smem + C::kQOff + x * C::kOperand + (warp & 3) * 4 * kOctet;
      auto raw = [&](int o, int k) { return operand + o * kOctet + (32 * (C::kWideK ? k : k & 1) + lane) * 16 + (k >> 1) * (C::kWideK ? 0 : C::kOperand / 2); };
#pragma unroll 1
      for (int o = 0; o < 4; ++o) {
        const int off = __shfl_sync(0xffffffffu, row_off, 8 * o + row);
        const __nv_bfloat16* src = p.q + (tile_row + max(off, 0)) * D + at * 8;
#pragma unroll
        for (int k = 0; k < D / 32; ++k)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(raw(o, k))), "l"(src + 32 * k), "r"(off >= 0 ? 16 : 0) : "memory");
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll 1
      for (int o = 0; o < 4; ++o) {
        uint4 q[D / 32];
        uint32_t m = 0;
#pragma unroll
        for (int k = 0; k < D / 32; ++k) {
          q[k] = *reinterpret_cast<const uint4*>(raw(o, k));
          m = __vmaxu2(m, __vmaxu2(__vmaxu2(q[k].x & 0x7FFF7FFFu, q[k].y & 0x7FFF7FFFu), __vmaxu2(q[k].z & 0x7FFF7FFFu, q[k].w & 0x7FFF7FFFu)));
        }
        m = __vmaxu2(m, __shfl_xor_sync(0xffffffffu, m, 8));
        m = __vmaxu2(m, __shfl_xor_sync(0xffffffffu, m, 16));
        const uint32_t amax = max(m << 16, m & 0xFFFF0000u);             // |bf16| as fp32 bits
        // the row scaled by a power of two into [128, 256), undone on the logits
        int k2 = 0;
        if (amax != 0u) k2 = max(-64, min(64, 134 - static_cast<int>((amax >> 23) & 0xFF)));
        // (and by the logits' sign: their scale is not negative from here on)
        const float up = copysignf(__uint_as_float(static_cast<uint32_t>(k2 + 127) << 23), p.sm_scale_log2);
        const float down = __shfl_sync(0xffffffffu, fabsf(p.sm_scale_log2) * __uint_as_float(static_cast<uint32_t>(127 - k2) << 23), row);
        if (at == o) qscale = down;
        __syncwarp();
#pragma unroll
        for (int k = 0; k < D / 32; ++k) {                // eight elements
          const uint32_t w[4] = {q[k].x, q[k].y, q[k].z, q[k].w};
          uint32_t h[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) h[e] = pack_f16x2(bf16_lo(w[e]) * up, bf16_hi(w[e]) * up);
          uint8_t* dst = operand + o * kOctet + row * 16;
          if constexpr (C::kWideK) {
            *reinterpret_cast<uint4*>(dst + (at + 4 * k) * 128) = make_uint4(h[0], h[1], h[2], h[3]);      // f16 (exact)
          } else {
            // the exact sum of the nearest E4M3 value and the E4M3 value of the remainder
            uint32_t lead[4], rest[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) { lead[e] = e4m3_term(h[e], 1.0f); rest[e] = f16x2_to_e4m3x2(h[e]); }
            dst += ((at + 4 * k) >> 1) * 128 + (at & 1) * 8;
            *reinterpret_cast<uint2*>(dst) = make_uint2(lead[0] | (lead[1] << 16), lead[2] | (lead[3] << 16));
            *reinterpret_cast<uint2*>(dst + C::kOperand / 2) = make_uint2(rest[0] | (rest[1] << 16), rest[2] | (rest[3] << 16));
          }
        }
      }
    }
    fence_proxy_async();
    __syncwarp();
    arrive_one(bar_q);

    // index of the last visible key of the row.  Rows past the tile's last query (their operand is zero, and they are never
    // stored) see everything, so that their warp takes the same unmasked path as its live rows.
    const int lim = live ? (p.causal ? min(L - 1, L - n_new + q0 + x * TQ + qi) : L - 1) : (1 << 30);
    const int halves = (tile_keys(x) + kHalf - 1) / kHalf, other_halves = (tile_keys(1 - x) + kHalf - 1) / kHalf;
    float m_ref = -INFINITY, m_use = 0.0f, l_row = 0.0f, v_ref = 0.0f;      // m_use: m_ref, or 0 before the first visible key
    bool ok = true;
#pragma unroll 1
    for (int h = 0; h < halves && ok; ++h) {
      const int t = h >> 1, buf = h & 1;
      const float* sc = scales + (t & (C::kScaleSlots - 1)) * 32 + 4 * buf;
      ok = wait_warp(&bar_sfull[2 * x + buf], t & 1u, abort_flag);
      if (!ok) break;
      tc_fence_after();
      uint32_t s[2][32];
#pragma unroll
      for (int i = 0; i < 2; ++i) tmem_ld32_issue(s_cols + kHalf * buf + 32 * i, s[i]);
      const float4 sk = *reinterpret_cast<const float4*>(sc), lg = *reinterpret_cast<const float4*>(sc + 8), inv = *reinterpret_cast<const float4*>(sc + 16);
      const float v_factor = buf == 0 ? sc[24] : 1.0f;
      // logit = accumulator * cf of its block (a zero scale: tiny, so that -inf stays -inf; none is negative)
      const float cf[4] = {fmaxf(sk.x * qscale, 1e-30f), fmaxf(sk.y * qscale, 1e-30f), fmaxf(sk.z * qscale, 1e-30f), fmaxf(sk.w * qscale, 1e-30f)};
#pragma unroll
      for (int i = 0; i < 2; ++i) tmem_ld_wait32(s[i]);
      const int visible = lim - h * kHalf;
      if (visible < kHalf - 1) {
#pragma unroll
        for (int j = 0; j < kHalf; ++j) s[j >> 5][j & 31] = j <= visible ? s[j >> 5][j & 31] : 0xFF800000u;      // -inf
      }
      float m_tile = -INFINITY;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const uint32_t* v = &s[c >> 1][(c & 1) * 16];
        auto f = [&](int j) { return __uint_as_float(v[j]); };
        const float m0 = max3(f(0), f(1), f(2)), m1 = max3(f(3), f(4), f(5)), m2 = max3(f(6), f(7), f(8)), m3 = max3(f(9), f(10), f(11)), m4 = max3(f(12), f(13), f(14));
        m_tile = fmaxf(m_tile, fmaxf(max3(m0, m1, m2), max3(m3, m4, f(15))) * cf[c]);
      }
      // lazy references: moved only when the half would push a probability (or a scale ratio) past the margin, so that the common
      // way through a half is one vote
      const bool move = m_tile > m_ref + kMaxLag;       // also true for the row's first visible key
      if (__any_sync(0xffffffffu, move || v_factor != 1.0f)) {
        float factor = v_factor;
        if (v_factor != 1.0f) v_ref = sc[25];
        if (move) {
          const float f = m_ref == -INFINITY ? 0.0f : ex2(m_ref - m_tile);
          factor *= f;
          l_row *= f;
          m_ref = m_use = m_tile;
        }
        if (h > 0) {
          // the accumulator is at rest once the product of the half before is done
          ok = wait_warp(&bar_pv[x], (h - 1) & 1u, abort_flag);
          if (!ok) break;
          tc_fence_after();
#pragma unroll 1
          for (int i = 0; i < D; i += 64) {
            uint32_t o[4][16];
#pragma unroll
            for (int e = 0; e < 4; ++e) tmem_ld16_issue(o_cols + i + 16 * e, o[e]);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              tmem_ld_wait(o[e]);
#pragma unroll
              for (int j = 0; j < 16; ++j) o[e][j] = __float_as_uint(__uint_as_float(o[e][j]) * factor);
              tmem_st16(o_cols + i + 16 * e, o[e]);
            }
          }
        }
      }
      // The two softmax warps of a scheduler take turns at the exponentials: tile 1's half h comes behind tile 0's h - 1, tile 0's
      // behind tile 1's h, as long as the other tile has such a half.  Side by side they would each take twice as long, and then
      // leave the units idle while both load logits and look for the maximum.  Tile 1 goes first because, if one of them has
      // more keys, it is that one.  (Tile 0 first / tile 1: 24 x 100..300 tokens, 8 heads, 41.3 / 40.6 us; 24 x 335..671 86.2 /
      // 85.0; four of 1000..2000, 40 over 8, 153.8 / 152.7; where the tiles are long and alike the same.)
      const int turn = x == 1 ? h - 1 : h;
      if (kTurns && turn >= 0 && turn < other_halves) ok = wait_warp(&bar_turn[4 * (1 - x) + (warp & 3)], turn & 1u, abort_flag);
      if (!ok) break;
      // p * pv = 2^(s * cf - m + log2 pv): the V scale rides in the exponent, and a block's sum of p is recovered from the sum
      // of p * pv (pv: the block's V scale over the reference, at most 2^4, a zero one replaced by 2^-24)
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        uint32_t pw[16];
#pragma unroll
        for (int e2 = 0; e2 < 2; ++e2) {
          const int c = 2 * i + e2;
          const float shift = (c == 0 ? lg.x : c == 1 ? lg.y : c == 2 ? lg.z : lg.w) - m_use;
          const uint32_t* v = &s[i][16 * e2];
          const uint64_t cf2 = f32_pair(cf[c], cf[c]), shift2 = f32_pair(shift, shift);
          uint64_t y[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const float2 t = f32_both(fma2(f32_pair(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1])), cf2, shift2));
            const float2 q = make_float2(ex2(t.x), ex2(t.y));
            pw[8 * e2 + e] = pack_f16x2(q.x, q.y);
            y[e] = f32_pair(q.x, q.y);
          }
          // (Summed as a tree: a chain of sums kept the exponentials waiting, 820-1040 cycles a half for one warp of a scheduler
          // against 590, with 512 that the exponentials need.)
          const float2 u = f32_both(add2(add2(add2(y[0], y[1]), add2(y[2], y[3])), add2(add2(y[4], y[5]), add2(y[6], y[7]))));
          l_row += (u.x + u.y) * (c == 0 ? inv.x : c == 1 ? inv.y : c == 2 ? inv.z : inv.w);
        }
        if (kTurns && i == 1) arrive_one(&bar_turn[4 * x + (warp & 3)]);       // (ahead of the store: behind it 394 us, here 385)
        tmem_st16(s_cols + kHalf * buf + 16 * i, pw);
      }
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      arrive_one(&bar_pfull[2 * x + buf]);
    }
    const bool any_keys = halves > 0;
    if (ok && any_keys) ok = wait_bar(&bar_out[x], 0u, abort_flag);
    ok = __all_sync(0xffffffffu, ok);
    if (ok) {
      tc_fence_after();
      const float k = l_row > 0.0f ? v_ref / l_row : 0.0f;
      // The rows go through shared memory, where the tile's query operand was (its products are done): 16 bytes of a row at
      // (chunk ^ row).
      constexpr int kLanes = D / 8, kRowsAt = 32 / kLanes;  // lanes of a row, rows at a time
      const int at = lane % kLanes, at_row = lane / kLanes;
      uint8_t* rows = smem + C::kQOff + x * C::kOperand + (warp & 3) * 32 * D * 2;
#pragma unroll 1
      for (int c = 0; c < D / 32; ++c) {
        uint32_t o[32];
        if (any_keys) {
          tmem_ld32_issue(o_cols + 32 * c, o);
          tmem_ld_wait32(o);
        }
        uint32_t w[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) w[j] = k != 0.0f ? pack_bf16x2(__uint_as_float(o[2 * j]) * k, __uint_as_float(o[2 * j + 1]) * k) : 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j)
          *reinterpret_cast<uint4*>(rows + lane * D * 2 + ((4 * c + j) ^ (lane & (kLanes - 1))) * 16) = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
      }
      __syncwarp();
#pragma unroll 4
      for (int i = 0; i < kLanes; ++i) {
        const int row = kRowsAt * i + at_row, off = __shfl_sync(0xffffffffu, row_off, row);
        if (off >= 0)
          *reinterpret_cast<uint4*>(p.out + (tile_row + off) * D + at * 8) = *reinterpret_cast<const uint4*>(rows + row * D * 2 + (at ^ (row & (kLanes - 1))) * 16);
      }
      tc_fence_before();
    } else if (lane == 0) {
      atomicCAS(p.status, 0, COOPT_ERR_TIMEOUT);
    }
  } else if (warp < kMmaWarp) {
    // ================= widening ==========================================================================================
    asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");
    const int wt = tid - kWidenWarp * 32;
    bool ok = true;
#pragma unroll 1
    for (int t = 0; t < n_tiles && ok; ++t) {
      const int w2 = t % C::kWide;
      const uint32_t w_use = t / C::kWide;
      const int nb = min(kTileBlocks, n_blocks - t * kTileBlocks);
      if constexpr (C::kWideK) {
        const int ks = t % C::kKSlots;
        ok = wait_bar(&bar_kfull[ks], (t / C::kKSlots) & 1u, abort_flag);
        if (ok && w_use > 0) ok = wait_bar(&bar_k16free[w2], (w_use - 1) & 1u, abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        // 16 dims of a token at a time: token (wt & 7) of an 8-token group, dims 16 c ..
        const uint8_t* src = smem + C::kKOff + ks * C::kKSlot;
        uint8_t* dst = smem + C::kK16Off + w2 * C::kOperand;
#pragma unroll 1
        for (int i = wt; i < nb * D; i += 128) {
          const int tok = i & 7, c = (i >> 3) % (D / 16), grp = (i >> 3) / (D / 16);
          const uint4 v = *reinterpret_cast<const uint4*>(src + grp * 8 * D + c * 128 + tok * 16);
          const uint2 a = widen4<kE5m2>(v.x), e = widen4<kE5m2>(v.y), f = widen4<kE5m2>(v.z), h = widen4<kE5m2>(v.w);
          uint8_t* to = dst + grp * 16 * D + c * 256 + tok * 16;
          *reinterpret_cast<uint4*>(to) = make_uint4(a.x, a.y, e.x, e.y);
          *reinterpret_cast<uint4*>(to + 128) = make_uint4(f.x, f.y, h.x, h.y);
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) { mbar_arrive(&bar_k16full[w2]); mbar_arrive(&bar_kfree[ks]); }
      }
      const int vs = t % C::kVSlots;
      ok = wait_bar(&bar_vfull[vs], (t / C::kVSlots) & 1u, abort_flag);
      if (ok && w_use > 0) ok = wait_bar(&bar_v16free[w2], (w_use - 1) & 1u, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      // dim d of V^T, the 16 tokens of a block at a time
      const int d = wt & (D - 1);
      const uint8_t* src = smem + C::kVOff + vs * C::kCodes + (d >> 3) * 128 + (d & 7) * 16;
      uint8_t* dst = smem + C::kV16Off + w2 * C::kOperand + (d >> 3) * 2048 + (d & 7) * 16;
      const int nkeys = kv_end - t * kTileKeys;
#pragma unroll 1
      for (int c = wt / D; c < nb; c += 128 / D) {
        const uint4 v = *reinterpret_cast<const uint4*>(src + c * C::kPart);
        uint32_t w[4] = {v.x, v.y, v.z, v.w};
        const int keep = nkeys - c * kBlockSize;
        if (keep < kBlockSize) {                          // the context ends inside this block: codes past it are cleared
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int left = keep - 4 * j;
            w[j] &= left >= 4 ? 0xFFFFFFFFu : (left <= 0 ? 0u : (1u << (8 * left)) - 1u);
          }
        }
        const uint2 a = widen4<kE5m2>(w[0]), e = widen4<kE5m2>(w[1]), f = widen4<kE5m2>(w[2]), h = widen4<kE5m2>(w[3]);
        *reinterpret_cast<uint4*>(dst + 2 * c * 128) = make_uint4(a.x, a.y, e.x, e.y);
        *reinterpret_cast<uint4*>(dst + (2 * c + 1) * 128) = make_uint4(f.x, f.y, h.x, h.y);
      }
      fence_proxy_async();                                // the tensor core will read what this thread has just written
      __syncwarp();
      if (lane == 0) { mbar_arrive(&bar_v16full[w2]); mbar_arrive(&bar_vfree[vs]); }
    }
    if (!ok && lane == 0) atomicCAS(p.status, 0, COOPT_ERR_TIMEOUT);
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");
    if (warp < kCopyWarp) {
      // ================= matrix instructions of one tile =================================================================
      {
        const int mx = warp - kMmaWarp;
        uint64_t* k_full = C::kWideK ? bar_k16full : bar_kfull;
        uint64_t* k_free = C::kWideK ? bar_k16free : bar_kfree;
        constexpr int kSlots = C::kWideK ? C::kWide : C::kKSlots;
        constexpr int kSlotBytes = C::kWideK ? C::kOperand : C::kKSlot;
        constexpr uint32_t kRowGroup = C::kWideK ? 16 * D : 8 * D;       // bytes of eight rows of Q, K
        const uint64_t desc_k = umma_desc(smem_u32(smem + (C::kWideK ? C::kK16Off : C::kKOff)), 128, kRowGroup);
        const uint64_t desc_q = umma_desc(smem_u32(smem + C::kQOff + mx * C::kOperand), 128, kRowGroup);
        const uint64_t desc_v = umma_desc(smem_u32(smem + C::kV16Off), 128, 2048);
        const uint32_t s_cols = tmem + 2 * kHalf * mx, o_cols = tmem + 4 * kHalf + D * mx;
        const int keys = tile_keys(mx), halves = (keys + kHalf - 1) / kHalf, my_tiles = (keys + kTileKeys - 1) / kTileKeys;
        bool ok = true;
        int done = 0;                                     // halves whose product with V has been seen to be done
        auto see_products = [&](int upto) {
          for (; ok && done < upto; ++done) {
            ok = wait_warp(&bar_pv[mx], done & 1u, abort_flag);
            if (ok && ((done & 1) || done == halves - 1)) arrive_one(&bar_v16free[(done >> 1) % C::kWide]);
          }
        };
        // Logits of a half, where those of half h - 2 and then its probabilities were: its product is done.
        auto issue_logits = [&](int h) {
          const int t = h >> 1, ks = t % kSlots;
          if ((h & 1) == 0) {
            ok = ok && wait_warp(&bar_scale[t & (C::kScaleSlots - 1)], (t / C::kScaleSlots) & 1u, abort_flag);
            ok = ok && wait_warp(&k_full[ks], (t / kSlots) & 1u, abort_flag);
          }
          if (!ok) return;
          tc_fence_after();
          const uint64_t dk = desc_k + ((ks * kSlotBytes + (h & 1) * 8 * kRowGroup) >> 4);
          const uint32_t to = s_cols + kHalf * (h & 1);
          if constexpr (C::kWideK) {
#pragma unroll
            for (int k = 0; k < D / 16; ++k) umma_f16(to, desc_q + k * 16, dk + k * 16, umma_idesc(kHalf), k != 0);
          } else {
#pragma unroll
            for (int term = 0; term < 2; ++term)
#pragma unroll
              for (int k = 0; k < D / 32; ++k)
                umma_f8(to, desc_q + ((term * (C::kOperand / 2)) >> 4) + k * 16, dk + k * 16, umma_idesc(kHalf, 0, kE5m2 ? 1 : 0), (term | k) != 0);
          }
          umma_commit(&bar_sfull[2 * mx + (h & 1)]);
          arrive_one(&bar_sfull[2 * mx + (h & 1)]);
        };
        ok = wait_warp(bar_q, 0u, abort_flag);
        if (halves > 0) issue_logits(0);
        if (halves > 1) issue_logits(1);
        for (int h = 0; h < halves && ok; ++h) {
          const int t = h >> 1, w2 = t % C::kWide;
          if ((h & 1) == 0) ok = ok && wait_warp(&bar_v16full[w2], (t / C::kWide) & 1u, abort_flag);
          ok = ok && wait_warp(&bar_pfull[2 * mx + (h & 1)], t & 1u, abort_flag);
          if (!ok) break;
          if ((h & 1) || h == halves - 1) arrive_one(&k_free[t % kSlots]);      // probabilities are there, so the logits have been
          tc_fence_after();
          const uint64_t dv = desc_v + ((w2 * C::kOperand) >> 4) + (h & 1) * 64;
          const uint32_t from = s_cols + kHalf * (h & 1);
          const int nb = min(kTileBlocks / 2, n_blocks - h * (kTileBlocks / 2));      // 16 keys (one cache block) per instruction
          if (nb == kTileBlocks / 2) {
#pragma unroll
            for (int k = 0; k < kTileBlocks / 2; ++k) umma_f16_ts(o_cols, from + 8 * k, dv + k * 16, umma_idesc(D), (h | k) != 0);
          } else {
            for (int k = 0; k < nb; ++k) umma_f16_ts(o_cols, from + 8 * k, dv + k * 16, umma_idesc(D), (h | k) != 0);
          }
          umma_commit(&bar_pv[mx]);
          // (Products are seen one by one: a wait for a barrier's phase must not fall two phases behind.)
          see_products(h + 1);
          if (h + 2 < halves) issue_logits(h + 2);
        }
        if (ok) {
          tc_fence_after();
          tc_fence_before();
          arrive_one(&bar_out[mx]);
        }
        for (int t = my_tiles; t < n_tiles && ok; ++t) {  // no row of this tile sees these keys
          const int ks = t % kSlots, w2 = t % C::kWide;
          ok = wait_warp(&k_full[ks], (t / kSlots) & 1u, abort_flag);
          if (ok) arrive_one(&k_free[ks]);
          ok = ok && wait_warp(&bar_v16full[w2], (t / C::kWide) & 1u, abort_flag);
          if (ok) arrive_one(&bar_v16free[w2]);
        }
        if (!ok && lane == 0) atomicCAS(p.status, 0, COOPT_ERR_TIMEOUT);
      }
    } else if (warp == kCopyWarp) {
      // ================= copies: per tile six gather requests of four granules' K parts, V parts or headers =============
      // Lane 3 q + w (q = 0, 1; w = 0, 1, 2) fetches the K parts (w = 0), the V parts (w = 1) or the headers (w = 2) of
      // granules 4 q .. 4 q + 3 of the tile.  Rows past the last block repeat the tile's first one.  The physical blocks are
      // looked up 32 at a time (four tiles, one per lane), a batch ahead of their use (range-checked: a bad id is reported in
      // the status word and replaced by block 0, never dereferenced).
      bool ok = true;
      const int q4 = lane / 3, what = lane - 3 * q4;
      const int col = what * (C::kPart / 8);
      const CUtensorMap* map = what == 2 ? &map_hdr : &map_part;
      const int* trow = p.block_table + static_cast<size_t>(b) * p.max_blocks_per_seq;
      auto load_batch = [&](int lb) -> int {
        const int j = lb * 32 + lane;
        int id = j < n_blocks ? trow[j] : 0;
        if (id < 0 || id >= p.num_blocks) { atomicCAS(p.status, 0, COOPT_ERR_INVALID_ARG); id = 0; }
        return id;
      };
      int ids_cur = load_batch(0), ids_next = load_batch(1);
      for (int t = 0; t < n_tiles; ++t) {
        const int nb = min(kTileBlocks, n_blocks - t * kTileBlocks);
        const int ngroups = (nb + 3) / 4;
        if (t > 0 && (t & 3) == 0) { ids_cur = ids_next; ids_next = load_batch((t >> 2) + 1); }
        int rows[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int j = (q4 & 1) * 4 + i;                           // block of the tile (lanes past the six copy lanes fetch along)
          rows[i] = __shfl_sync(0xffffffffu, ids_cur, (t & 3) * 8 + (j < nb ? j : 0)) * Hkv + g;
        }
        const int ks = t % C::kKSlots, vs = t % C::kVSlots;
        const uint32_t k_use = t / C::kKSlots, v_use = t / C::kVSlots;
        if (lane == 0) {
          if (k_use > 0) ok = wait_bar(&bar_kfree[ks], (k_use - 1) & 1u, abort_flag);
          if (ok) {
            mbar_expect_tx(&bar_kfull[ks], ngroups * 4 * (C::kPart + kFp8Header));
            pend_mask |= 1u << ks;
            pend_par = (pend_par & ~(1u << ks)) | ((k_use & 1u) << ks);
          }
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
        if (!ok) break;
        __syncwarp();                                     // what lane 0 has waited for holds for the lanes that copy
        if (lane < 3 * ngroups && what != 1)
          gather4_g2s(smem + C::kKOff + ks * C::kKSlot + (what == 2 ? C::kCodes + q4 * 4 * kFp8Header : q4 * 4 * C::kPart), map, col, rows[0], rows[1], rows[2], rows[3], &bar_kfull[ks]);
        if (lane == 0) {
          if (v_use > 0) ok = wait_bar(&bar_vfree[vs], (v_use - 1) & 1u, abort_flag);
          if (ok) {
            mbar_expect_tx(&bar_vfull[vs], ngroups * 4 * C::kPart);
            pend_mask |= 16u << vs;
            pend_par = (pend_par & ~(16u << vs)) | ((v_use & 1u) << (4 + vs));
          }
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
        if (!ok) break;
        __syncwarp();                                     // what lane 0 has waited for holds for the lanes that copy
        if (lane < 3 * ngroups && what == 1)
          gather4_g2s(smem + C::kVOff + vs * C::kCodes + q4 * 4 * C::kPart, map, col, rows[0], rows[1], rows[2], rows[3], &bar_vfull[vs]);
      }
      if (!ok && lane == 0) atomicCAS(p.status, 0, COOPT_ERR_TIMEOUT);
    } else {
      // ================= block scales, as the softmax uses them =============================================================
      float v_ref = 0.0f;
      bool ok = true;
      for (int t = 0; t < n_tiles; ++t) {
        const int ks = t % C::kKSlots;
        ok = wait_bar(&bar_kfull[ks], (t / C::kKSlots) & 1u, abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        const int nb = min(kTileBlocks, n_blocks - t * kTileBlocks);
        float sk = 0.0f, sv = 0.0f;
        if (lane < nb) {
          const float2 h = *reinterpret_cast<const float2*>(smem + C::kKOff + ks * C::kKSlot + C::kCodes + lane * kFp8Header);
          sk = h.x; sv = h.y;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar_kfree[ks]);
        const float v_tile = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(sv)));   // scales are not negative
        float factor = 1.0f;
        if (v_tile > v_ref * kScaleLag) {
          factor = v_ref > 0.0f ? v_ref / v_tile : 0.0f;
          v_ref = v_tile;
        }
        // (a slot is free again four tiles on: the K slots behind its tile's are handed out only once these scales have been used)
        float* sc = scales + (t & (C::kScaleSlots - 1)) * 32;
        const float pv = fmaxf(v_ref > 0.0f ? sv / v_ref : 0.0f, 0x1p-24f);
        if (lane < kTileBlocks) {
          float lg;
          asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(lg) : "f"(pv));
          sc[lane] = sk;
          sc[8 + lane] = lg;
          sc[16 + lane] = 1.0f / pv;
          if (lane == 0) { sc[24] = factor; sc[25] = v_ref; }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar_scale[t & (C::kScaleSlots - 1)]);
      }
      if (!ok && lane == 0) atomicCAS(p.status, 0, COOPT_ERR_TIMEOUT);
    }
  }

  // ---- exit: copies still in flight get a bounded time to land, tensor memory is returned -----------
  __syncthreads();
  if (*abort_flag != 0 && warp == kCopyWarp && lane == 0) {
    for (int i = 0; i < C::kKSlots; ++i)
      if ((pend_mask >> i) & 1u) mbar_wait_bounded(&bar_kfull[i], (pend_par >> i) & 1u);
    for (int i = 0; i < C::kVSlots; ++i)
      if ((pend_mask >> (4 + i)) & 1u) mbar_wait_bounded(&bar_vfull[i], (pend_par >> (4 + i)) & 1u);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

template <int D, bool kE5m2>
int launch_one(const coopt_cache* c, const PrefillParams& p, dim3 grid, cudaStream_t stream) {
  using C = Cfg<D>;
  CUtensorMap map_part, map_hdr;
  const long long granules = static_cast<long long>(c->num_blocks) * c->num_kv_heads;
  if (!encode_cache_map(&map_part, c->data, granules, C::kGran, C::kPart / 8) || !encode_cache_map(&map_hdr, c->data, granules, C::kGran, kFp8Header / 8))
    return COOPT_ERR_CUDA;
  auto launch = [&](auto* kernel) {
    if (!configure_kernel_smem(reinterpret_cast<const void*>(kernel), C::kSmemBytes)) return COOPT_ERR_CUDA;
    return launch_dependent(kernel, grid, kThreads, C::kSmemBytes, stream, p, map_part, map_hdr) ? COOPT_OK : COOPT_ERR_CUDA;
  };
  return p.tiles == 2 ? launch(&paged_prefill_kernel<D, kE5m2, true>) : launch(&paged_prefill_kernel<D, kE5m2, false>);
}

}  // namespace

int launch_paged_prefill(const coopt_cache* c, const void* q, void* out, const int32_t* cu_q_lens,
                         const int32_t* block_table, int32_t max_blocks_per_seq, const int32_t* context_lens,
                         int32_t batch, int32_t num_q_heads, int32_t total_q, int32_t causal, float sm_scale,
                         void* workspace, int num_sms, cudaStream_t stream) {
  if (!is_fp8(c->dtype)) return COOPT_ERR_UNSUPPORTED;
  if (c->dtype == COOPT_KV_FP8_E5M2 && c->head_dim != 128) return COOPT_ERR_UNSUPPORTED;
  PrefillParams p;
  p.q = static_cast<const __nv_bfloat16*>(q);
  p.out = static_cast<__nv_bfloat16*>(out);
  p.cu_q_lens = cu_q_lens;
  p.block_table = block_table;
  p.context_lens = context_lens;
  p.max_blocks_per_seq = max_blocks_per_seq;
  p.batch = batch;
  p.num_q_heads = num_q_heads;
  p.num_kv_heads = c->num_kv_heads;
  p.group = num_q_heads / c->num_kv_heads;
  p.num_blocks = c->num_blocks;
  p.tile_queries = kRows / p.group;
  p.causal = causal;
  p.sm_scale_log2 = sm_scale * kLog2e;
  p.status = static_cast<int*>(workspace);
  auto most = [&](int tiles) { return static_cast<long long>(total_q) / (tiles * p.tile_queries) + batch; };   // every sequence adds at most one that is partly filled
  // A CTA with one tile takes about 0.73 of the time of one with two (the tensor core and the exponential units are less busy,
  // and so nothing waits as long), but twice as many are needed: one tile as long as all of them start at once.  (One sequence,
  // 40 heads over 8, head_dim 128: 256 new tokens behind 8000 139.5 us with two / 108.6 with one, 512 behind 8000, which
  // would be 168 CTAs, 151 with two; 8 heads over 1, 128 behind 32000 508 / 370, 2048 alone 42.1 / 32.6.)
  p.tiles = most(1) * c->num_kv_heads <= num_sms ? 1 : 2;
  const long long pairs = most(p.tiles);
  if (pairs * c->num_kv_heads > 0x7fffffffll) return COOPT_ERR_UNSUPPORTED;
  const dim3 grid(static_cast<unsigned>(pairs * c->num_kv_heads));
  p.by_length = pairs * c->num_kv_heads > num_sms ? 1 : 0;
  if (c->head_dim == 64) return launch_one<64, false>(c, p, grid, stream);
  return c->dtype == COOPT_KV_FP8_E5M2 ? launch_one<128, true>(c, p, grid, stream) : launch_one<128, false>(c, p, grid, stream);
}

}  // namespace coopt
