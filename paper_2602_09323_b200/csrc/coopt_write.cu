// coopt_kv_write: Opt-KV cache write (Algorithm 1 phase 1, Eq. 5) with per-(block, kv head)
// dynamic FP8 E4M3 scales.  One warp owns one (token group, kv head): it is the only writer of
// that granule during the call, so the scale update and the re-expression of resident codes
// need no atomics.
#include "coopt_write.cuh"

namespace coopt {

namespace {

constexpr int kWriteHeads = 4;                 // kv heads per CTA
constexpr int kWriteWarps = 2 * kWriteHeads;   // FP8: one warp per (kv head, K | V)

// FP8, few tokens (decode steps): one CTA per (token, kWriteHeads kv heads), one warp per
// (kv head, K | V); CTAs whose token leads no group leave at once.
template <int D, bool kE5m2>
__global__ void __launch_bounds__(kWriteWarps * 32) kv_write_fp8_kernel(WriteParams p) {
  __shared__ __align__(16) uint8_t stage[kWriteWarps][part_bytes(D, true)];
  __shared__ Group group;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  wait_previous_kernel();
  if (warp == 0) find_group_warp(p, blockIdx.x, group, lane);
  __syncthreads();
  if (group.n == 0) return;
  const int h = blockIdx.y * kWriteHeads + (warp >> 1);
  if (h >= p.num_kv_heads) return;
  write_part<D, kE5m2>(p, group, h, warp & 1, stage[warp], lane);
}

// The K part (which = 0) or the V part (which = 1) of a block that is written whole: its 16 tokens follow one another in the
// call from `tok` on, in order, rows aligned for the loads below.  The same scale rule and the same value for every number
// that is stored as write_part (which takes the blocks that are not whole).  One warp; lane l has dims l D/32 .. of all 16
// tokens in registers.  K goes through shared memory (st, 16 D bytes; 16-byte pieces swizzled so that neither side meets a
// bank twice) and leaves as whole lines, V is in order in registers and leaves as 32-byte pieces.
// False if the scale is outside of the range that the reciprocal serves: nothing has been written then.
template <int D, bool kE5m2>
__device__ __forceinline__ bool write_whole_part(const WriteParams& p, int blk, int tok, int h, int which, uint8_t* st, int lane) {
  constexpr int kPart = part_bytes(D, true), kPerLane = D / 32, kWords = kPerLane / 2;
  uint32_t raw[kBlockSize][kWords];
  const __nv_bfloat16* row = (which == 0 ? p.k : p.v) + static_cast<int64_t>(tok) * p.token_stride + h * D + lane * kPerLane;
#pragma unroll
  for (int t = 0; t < kBlockSize; ++t) load_row<kPerLane, true>(row + t * p.token_stride, raw[t]);
  uint32_t top = 0;
#pragma unroll
  for (int t = 0; t < kBlockSize; ++t)
#pragma unroll
    for (int e = 0; e < kWords; ++e) asm("max.xorsign.abs.bf16x2 %0, %0, %1;" : "+r"(top) : "r"(raw[t][e]));
  // (magnitudes of bf16 values order like their patterns)
  const uint32_t am = __reduce_max_sync(0xffffffffu, max((top << 16) & 0x7FFFFFFFu, top & 0x7FFF0000u));
  const float s = __fdiv_rn(__uint_as_float(am), kE5m2 ? kE5m2Max : kE4m3Max);
  if (!(s >= 0x1p-40f && s <= 0x1p40f)) return false;
  // x / s, correctly rounded (Markstein: r = RN(1 / s), q0 = RN(x r), RN(q0 + (x - s q0) r)).  With the residual taken as
  // s q0 - x a zero keeps the sign of x.
  const float r = __frcp_rn(s);
  auto quotient = [&](int t, int e) -> float {
    const float x = (e & 1) ? bf16_hi(raw[t][e >> 1]) : bf16_lo(raw[t][e >> 1]);
    const float q0 = __fmul_rn(x, r);
    return __fmaf_rn(-__fmaf_rn(s, q0, -x), r, q0);
  };
  uint8_t* gran = p.cache + (static_cast<size_t>(blk) * p.num_kv_heads + h) * granule_bytes(D, true);
  uint8_t* part = gran + which * kPart;
  if (which == 0) {
    constexpr int kChunks = D / 16;                       // 16-byte pieces of a token
    auto place = [&](int t, int c) { return t * D + (c ^ (D == 128 ? t & 7 : (t >> 1) & 3)) * 16; };
#pragma unroll
    for (int t = 0; t < kBlockSize; ++t) {
      uint8_t* dst = st + place(t, lane * kPerLane / 16) + lane * kPerLane % 16;
      if constexpr (kPerLane == 4)
        *reinterpret_cast<uint32_t*>(dst) = f32x2_to_codes<kE5m2>(quotient(t, 0), quotient(t, 1)) | (f32x2_to_codes<kE5m2>(quotient(t, 2), quotient(t, 3)) << 16);
      else
        *reinterpret_cast<uint16_t*>(dst) = static_cast<uint16_t>(f32x2_to_codes<kE5m2>(quotient(t, 0), quotient(t, 1)));
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < kPart / 512; ++i) {
      const int o = i * 32 + lane, t = (o / (8 * kChunks)) * 8 + (o & 7), c = (o >> 3) % kChunks;
      reinterpret_cast<uint4*>(part)[o] = *reinterpret_cast<const uint4*>(st + place(t, c));
    }
    __syncwarp();                                         // (the staging area may be written again)
  } else {
#pragma unroll
    for (int e = 0; e < kPerLane; e += 2) {               // two dims: 2 x 16 bytes in a row
      uint32_t w[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int d = e + (k >> 2), t = 4 * (k & 3);
        w[k] = f32x2_to_codes<kE5m2>(quotient(t, d), quotient(t + 1, d)) | (f32x2_to_codes<kE5m2>(quotient(t + 2, d), quotient(t + 3, d)) << 16);
      }
      asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(part + (lane * kPerLane + e) * 16), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]),
                   "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
    }
  }
  float* header = reinterpret_cast<float*>(gran + header_offset(D));
  if (lane == 0) header[which] = s;
  if (which == 0 && lane < 6) header[2 + lane] = 0.0f;
  return true;
}

// FP8, many tokens (prefill chunks, bulk fills): one CTA (kShared: several) per (kSpan consecutive tokens, kWriteHeads kv
// heads), a warp per (kv head, K | V).  Every warp finds the span's groups by itself: no warp waits for another.
// Bound by memory: 65,536 tokens of 8 heads x 128 (403 MB) in 65.9 us, 6.1 TB/s.  Before blocks written whole had a path of
// their own it was 112.6 us, bound by the integer pipe (10.6 instructions a value: look-ups of rows and groups, signs put
// back after the division, stores of K words eight lanes to a bank).
constexpr int kSpan = 32;
constexpr int kSpanThreshold = 512;     // calls with more tokens than this take the span kernel
// Groups that are not whole blocks take a warp 2 us each, one after the other (head_dim 128: the kernel's registers are what
// whole blocks want).  Where spans are few, several CTAs share one: as many as bring the launch to 8 CTAs an SM (6 at head_dim
// 64, where a group is shorter), a power of two, kSpanSplit at most.  300 sequences of 2 tokens 41.1 -> 8.7 us, 128 of 7 28.5 ->
// 8.4, 300 of 7 29.2 -> 15.8, 300 of 13 tokens 19.8 -> 16.8 (with 6 CTAs an SM, which shares by two there, 23.5); calls whose
// spans are not shared have a kernel without the choice (30,000 tokens of one kv head 6.6 us, 6.8 with it).
constexpr int kSpanSplit = 16;
template <int D, bool kE5m2, bool kShared>
__global__ void __launch_bounds__(kWriteWarps * 32, 4) kv_write_fp8_span_kernel(WriteParams p) {
  __shared__ __align__(16) uint8_t stage[kWriteWarps][part_bytes(D, true)];
  __shared__ Group groups[kWriteWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int h = blockIdx.y * kWriteHeads + (warp >> 1), which = warp & 1;
  wait_previous_kernel();
  if (h >= p.num_kv_heads) return;
  // the slots of the span, of the token before it, and of the 32 tokens behind it
  const int base = blockIdx.x * kSpan;
  auto slot_of = [&](int i) -> int64_t { return i >= 0 && i < p.num_tokens ? p.slot_mapping[i] : -1; };
  const int64_t s0 = slot_of(base + lane), s1 = slot_of(base + 32 + lane), before = slot_of(base - 1);
  const int64_t s0_up = __shfl_up_sync(0xffffffffu, s0, 1), s0_last = __shfl_sync(0xffffffffu, s0, 31), s1_up = __shfl_up_sync(0xffffffffu, s1, 1);
  const int64_t s0_prev = lane == 0 ? before : s0_up, s1_prev = lane == 0 ? s0_last : s1_up;
  // bit i: token base + i follows the token before it into the next offset of the same block
  const unsigned long long follows = __ballot_sync(0xffffffffu, s0 >= 0 && s0_prev >= 0 && s0 == s0_prev + 1 && (s0 % kBlockSize) != 0) |
                                     static_cast<unsigned long long>(__ballot_sync(0xffffffffu, s1 >= 0 && s1_prev >= 0 && s1 == s1_prev + 1 && (s1 % kBlockSize) != 0)) << 32;
  const bool begins = s0 >= 0 && s0 % kBlockSize == 0 && s0 / kBlockSize < p.num_blocks;
  // a block written whole begins with its first slot and 15 tokens follow it in order (the precondition of the call, a
  // block's tokens being consecutive, leaves no other token of it)
  unsigned whole = __ballot_sync(0xffffffffu, begins && ((follows >> (lane + 1)) & 0x7FFFull) == 0x7FFFull);
  // tokens that may lead any other group: all that do not follow into a block (a skipped token may stand between them and
  // the one they follow: find_group_warp looks closer)
  unsigned others = __ballot_sync(0xffffffffu, s0 >= 0 && !((follows >> lane) & 1ull)) & ~whole;
  const bool aligned = ((reinterpret_cast<uintptr_t>(which == 0 ? p.k : p.v) | static_cast<uintptr_t>(p.token_stride * 2)) & (D / 16 - 1)) == 0;
  if (!aligned) { others |= whole; whole = 0; }
  if constexpr (kShared) {                 // this CTA's part of the span's groups
    const unsigned mine = __ballot_sync(0xffffffffu, (__popc((whole | others) & ((1u << lane) - 1u)) & (gridDim.z - 1)) == blockIdx.z);
    whole &= mine;
    others &= mine;
  }
  while (whole) {
    const int w = __ffs(whole) - 1;
    whole &= whole - 1;
    const int blk = static_cast<int>(__shfl_sync(0xffffffffu, s0, w) / kBlockSize);
    if (!write_whole_part<D, kE5m2>(p, blk, base + w, h, which, stage[warp], lane)) others |= 1u << w;
  }
  while (others) {
    const int w = __ffs(others) - 1;
    others &= others - 1;
    find_group_warp(p, base + w, groups[warp], lane);
    __syncwarp();
    if (groups[warp].n > 0) write_part<D, kE5m2>(p, groups[warp], h, which, stage[warp], lane);
    __syncwarp();
  }
}

// bf16 ablation cache: store the values unchanged at their permuted places.
template <int D>
__global__ void __launch_bounds__(kWriteWarps * 32) kv_write_bf16_kernel(WriteParams p) {
  constexpr int kPerLane = D / 32;
  wait_previous_kernel();
  const int i = blockIdx.x;
  const int64_t slot = p.slot_mapping[i];
  if (slot < 0) return;                                   // Eq. 5
  const int64_t blk = slot / kBlockSize;
  if (blk >= p.num_blocks) return;
  const int off = static_cast<int>(slot % kBlockSize);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int h = blockIdx.y * kWriteWarps + warp;
  if (h >= p.num_kv_heads) return;
  uint8_t* gran = p.cache + (static_cast<size_t>(blk) * p.num_kv_heads + h) * granule_bytes(D, false);
#pragma unroll
  for (int which = 0; which < 2; ++which) {
    const __nv_bfloat16* row = (which == 0 ? p.k : p.v) + static_cast<int64_t>(i) * p.token_stride + h * D + lane * kPerLane;
    uint8_t* part = gran + part_offset(D, false, which);
#pragma unroll
    for (int e = 0; e < kPerLane; ++e) {
      const int d = lane * kPerLane + e;
      const int pos = which == 0 ? k_elem_offset(D, false, off, d) : v_elem_offset(D, false, off, d);
      *reinterpret_cast<__nv_bfloat16*>(part + pos) = row[e];
    }
  }
}

}  // namespace

int launch_kv_write(const coopt_cache* c, const void* k, const void* v, int64_t stride, const int64_t* slots,
                    int num_tokens, cudaStream_t stream) {
  WriteParams p;
  p.cache = static_cast<uint8_t*>(c->data);
  p.k = static_cast<const __nv_bfloat16*>(k);
  p.v = static_cast<const __nv_bfloat16*>(v);
  p.slot_mapping = slots;
  p.token_stride = stride;
  p.num_tokens = num_tokens;
  p.num_kv_heads = c->num_kv_heads;
  p.num_blocks = c->num_blocks;
  const bool fp8 = is_fp8(c->dtype), e5m2 = c->dtype == COOPT_KV_FP8_E5M2;
  // FP8: a CTA serves kWriteHeads kv heads (two warps each); bf16: kWriteWarps heads (one warp each)
  const int heads_per_cta = fp8 ? kWriteHeads : kWriteWarps;
  const int head_ctas = (c->num_kv_heads + heads_per_cta - 1) / heads_per_cta;
  const dim3 grid(num_tokens, head_ctas);
  const long long spans = (static_cast<long long>(num_tokens) + kSpan - 1) / kSpan * head_ctas;
  const DeviceInfo* di = device_info();
  int split = 1;
  while (2 * split <= kSpanSplit && 2 * split * spans <= (c->head_dim == 128 ? 8 : 6) * (di ? di->num_sms : 148)) split *= 2;
  const dim3 span_grid((num_tokens + kSpan - 1) / kSpan, head_ctas, split);
  const bool span = fp8 && num_tokens > kSpanThreshold;
  const auto launch = [&](auto kernel, dim3 ctas) { return launch_dependent(kernel, ctas, kWriteWarps * 32, 0, stream, p); };
  const auto launch_fp8 = [&](auto few, auto many, auto shared) { return !span ? launch(few, grid) : split > 1 ? launch(shared, span_grid) : launch(many, span_grid); };
  bool ok;
  if (c->head_dim == 128) {
    if (e5m2) ok = launch_fp8(kv_write_fp8_kernel<128, true>, kv_write_fp8_span_kernel<128, true, false>, kv_write_fp8_span_kernel<128, true, true>);
    else if (fp8) ok = launch_fp8(kv_write_fp8_kernel<128, false>, kv_write_fp8_span_kernel<128, false, false>, kv_write_fp8_span_kernel<128, false, true>);
    else ok = launch(kv_write_bf16_kernel<128>, grid);
  } else {
    if (e5m2) ok = launch_fp8(kv_write_fp8_kernel<64, true>, kv_write_fp8_span_kernel<64, true, false>, kv_write_fp8_span_kernel<64, true, true>);
    else if (fp8) ok = launch_fp8(kv_write_fp8_kernel<64, false>, kv_write_fp8_span_kernel<64, false, false>, kv_write_fp8_span_kernel<64, false, true>);
    else ok = launch(kv_write_bf16_kernel<64>, grid);
  }
  return ok ? COOPT_OK : COOPT_ERR_CUDA;
}

}  // namespace coopt
