// Paged GQA decode: Algorithm 1 phase 2 (Eq. 6 dequantisation on load), Algorithm 2 (Eq. 7-8: the G query heads of a
// group consume one K/V stream), Algorithm 3 (Eq. 9 valid blocks only, Eq. 10 max-subtracted softmax), the Opt-Pa
// chunk-and-merge reduction, and, in a step that appends, Algorithm 1 phase 1 for one token per sequence.  FP8 (E4M3,
// E5M2) and bf16 caches, head_dim 64 and 128, group sizes 1 to 8.
//
// What bounds it is the stream of the cache from HBM; everything else is arranged so that nothing waits on anything
// but that stream.  Every warp is on its own: it walks its part of the line of blocks (coopt_decode.cuh), a lane of it
// requests one granule (K part, V part, scales: one contiguous piece) per bulk copy into a ring of the warp's own, and
// the warp takes both contractions of a block from there as they land:
//     S^T [16 tokens x 8 heads] = K [16 x D] . Q^T        O^T [D x 8 heads] += V^T [D x 16 tokens] . P^T
// on mma.sync m16n8k16.  Tokens (and dims) fill the instruction's 16 rows and the heads of a group its 8 columns, so
// no row is idle for any group size.  Codes become f16 on the way from shared memory to registers (exact); a bf16
// query row, scaled by a power of two, is exact in f16 as well; a probability is f16 once, carried times 2^8 against a
// reference that may lag the maximum by 2^6, so that the running output is rescaled rarely; the K scale of a block
// multiplies its logits, the V scale goes into the probabilities.  No barrier is met between the first block and the
// last; pieces of units that warps or CTAs share are merged by log-sum-exp at the end.
//
// (On tcgen05.mma, 128 tokens at a time, the tensor core was 21 % busy with columns that are mostly padding, and the launch
// waited for hand-overs between its roles.  On tcgen05 / here: 24 sequences of 300..4000 tokens, G = 8, 46 / 23 us a layer;
// 32 x 2048 tokens, G = 5, 35 / 29; 64 sequences of 128..8192 tokens 121 / 104; 120 of 5..900, head_dim 64, 56 / 17.)
//
// A launch of 32 x 2048 tokens streams at 6.4 TB/s from its first copies, 3 us after a CTA's first instruction, to the end
// of its last block, 5 us before the CTA's last; code that runs once costs about four cycles an instruction to fetch.
// Registers are what the loop over blocks is short of: the walks of the copies and of the work wait in shared memory, and the
// query rows of a unit are fetched when it starts (eight layers of 21 sequences of 2..60 tokens: 49 / 43.6 us; prefetching the
// rows into registers at the end of the unit before instead: 49.5).
//
// (Two blocks at a time, contractions and exponentials side by side, each block by its own references, against one: eight layers
// of 32 x 2048 tokens 233 / 227 us, 64 of 128..8192, four layers, 411 / 404, four of 32768..131072 in chunks 127.5 / 125.8, 30 x
// 1597 34.5 / 32.1; only eight layers of 64 x 100..5000, head_dim 64, are a little faster, 174 / 176.)
#include <float.h>

#include <algorithm>

#include "coopt_decode.cuh"
#include "coopt_trace.cuh"
#include "coopt_umma.cuh"
#include "coopt_write.cuh"

namespace coopt {

namespace {

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr float kLag = 6.0f;                                      // how far a reference maximum may lag (base-2 logarithm units)
constexpr float kShift = 8.0f, kUnshift = 1.0f / 256.0f;          // probabilities are carried times 2^kShift: at most 2^14 in f16

constexpr int kMaxSmem = 232448;                                 // of a CTA

template <int D, int FMT>
struct Cfg {
  static constexpr bool kFp8 = FMT != COOPT_KV_BF16;
  [[maybe_unused]] static constexpr bool kE5m2 = FMT == COOPT_KV_FP8_E5M2;
  // A warp needs time for a block (about 1 us from landing to the next wait), so many warps are wanted, with two blocks in
  // flight each, or four of head_dim 64.  More of them in flight take longer: head_dim 128, 2 / 3 blocks 404 / 424 us (64
  // sequences of 128..8192 tokens, four layers), 125.8 / 133.0 (four of 32768..131072 in chunks), 219.5 / 228.3 (32 x 4096, four
  // launches), 226.6 / 227.6 (eight layers of 32 x 2048), 32.1 / 32.4 (30 x 1597); head_dim 64, 4 / 5: 138.6 / 139.8 (64 of
  // 100..5000, G = 4, four layers), 17.1 / 17.3 (120 of 5..900).  bf16: 8 x 2 and 8 x 4 (182 registers).
  static constexpr int kWarps = kFp8 ? (D == 128 ? 12 : 16) : 8;
  static constexpr int kThreads = kWarps * 32;
  static constexpr int kGran = granule_bytes(D, kFp8);
  static constexpr int kCopy = kFp8 ? 2 * kBlockSize * D + kFp8Header : kGran;   // bytes of a granule that are read
  static constexpr int kWholeIdle = kFp8 ? kWholeUnitsIdle : kWholeUnitsIdleBf16 * (D / 64);
  static constexpr int kPieceStride = D + 4;                    // floats of one head of a piece: o[D], maximum, sum, padding
  static constexpr int kPiece = kMaxGroup * kPieceStride * 4;   // bytes
  // A warp's shared memory: its ring, the piece of a unit from before, and, in a launch over several layers, the piece of a
  // unit that goes on (in a launch over one the ring has done its work by then, and the piece takes its place).
  static constexpr int kStages = D == 128 ? 2 : 4;
  static constexpr int kWarpBytes = kStages * kGran + (kFp8 ? 2 : 1) * kPiece;
  static constexpr int kBarOff = kWarps * kWarpBytes;
  static constexpr int kLensOff = kBarOff + (kWarps * kStages + 2) * 8;
  static constexpr int kPreOff = kLensOff + kMaxBatch * 4;
  static constexpr int kRecOff = kPreOff + (kMaxBatch + 4) * 4;
  static constexpr int kMiscOff = kRecOff + kWarps * 32;
  static constexpr int kCopyWalkOff = kMiscOff + 192;           // walks of a warp: where its copies are, and where its work is
  static constexpr int kSmemBytes = kCopyWalkOff + kWarps * 128;
  static_assert(kGran % 128 == 0 && kPiece % 128 == 0 && kStages * kGran >= kPiece && kWarpBytes % 128 == 0 && kCopy % 16 == 0, "copies land on 128-byte boundaries");
  static_assert(kStages >= 2 && kSmemBytes <= kMaxSmem, "room for copies in flight");
  static_assert(kCtasPerSm * (kSmemBytes + 1024) <= 233472, "shared memory of one SM");
};

// What a warp leaves about the (at most two) units it holds only a piece of.
struct Rec {
  int flags;            // kHas0: a piece of a unit that starts before this warp; kEnds0: that unit ends here; kHas1: one that starts here and goes on
  int b0, g0, u0;       // its sequence, kv head and first block
  int b1, g1, u1;
  int pad;
};
constexpr int kHas0 = 1, kEnds0 = 2, kHas1 = 4;
static_assert(sizeof(Rec) == 32, "shared memory layout");

// ---- the line ------------------------------------------------------------------------------------------------------
struct Line {
  const int* lens;      // shared memory: context lengths
  const unsigned* pre;  // shared memory: places of one kv head of the sequences before
  int batch, heads, chunk;   // chunk: blocks per chunk, kNoChunks without chunks
};
__device__ __forceinline__ int line_blocks(const Line& ln, int b) { return (ln.lens[b] + kBlockSize - 1) / kBlockSize; }
// first place of the unit of (b, g) that starts with block u
__device__ __forceinline__ unsigned unit_place(const Line& ln, int b, int g, int u) {
  const unsigned head = ln.pre[b + 1] - ln.pre[b];
  return ln.heads * ln.pre[b] + g * head + (ln.chunk == kNoChunks ? 0u : static_cast<unsigned>(u / ln.chunk) * static_cast<unsigned>(ln.chunk + kUnitCost));
}
__device__ __forceinline__ int unit_blocks(const Line& ln, int nb, int u) { return min(ln.chunk, nb - u); }

// A walk over the units of the places [x, end): unit (b, g, first block u, n blocks), of which the blocks [j, jend)
// (counted from u) belong to the walker.
constexpr int kSomeEmpty = 1 << 28;      // added to a warp's longest unit: a sequence's context is empty
struct Walk {
  int b, g, nb, u, n;
  int j, jend;
  unsigned base, end;
  int more;
  int pad[2];
};
static_assert(sizeof(Walk) == 48, "shared memory layout");
__device__ __forceinline__ void walk_range(Walk& w, unsigned x) {
  w.j = max(0, static_cast<int>(x - w.base) - kUnitCost);
  w.jend = min(w.n, static_cast<int>(w.end - w.base) - kUnitCost);
  w.more = w.jend > w.j;
}
__device__ __forceinline__ void walk_next(const Line& ln, Walk& w) {
  const unsigned at = w.base + w.n + kUnitCost;
  w.u += w.n;
  if (w.u >= w.nb) {
    w.u = 0;
    if (++w.g == ln.heads) {
      w.g = 0;
      ++w.b;
      while (w.b < ln.batch && ln.pre[w.b + 1] == ln.pre[w.b]) ++w.b;
      if (w.b >= ln.batch) { w.more = false; return; }
      w.nb = line_blocks(ln, w.b);
    }
  }
  w.base = at;
  w.n = unit_blocks(ln, w.nb, w.u);
  if (w.base >= w.end) { w.more = false; return; }
  walk_range(w, w.base);
}
// the sequence whose places contain x < all places (by the lanes of a warp together: 32 coarse candidates, then the fine ones)
__device__ __forceinline__ int line_seq(const Line& ln, unsigned x, int lane) {
  const int step = (ln.batch + 31) / 32;
  int c = lane * step;
  unsigned le = __ballot_sync(0xffffffffu, c < ln.batch && ln.heads * ln.pre[min(c, ln.batch)] <= x);
  const int lo = (31 - __clz(le)) * step;
  c = lo + lane;
  le = __ballot_sync(0xffffffffu, lane < step && c < ln.batch && ln.heads * ln.pre[min(c, ln.batch)] <= x);
  return lo + 31 - __clz(le);
}
// the unit that contains place x, and its first place
__device__ __forceinline__ void walk_unit(const Line& ln, Walk& w, unsigned x, int lane) {
  w.b = line_seq(ln, x, lane);
  const unsigned before = ln.heads * ln.pre[w.b], head = ln.pre[w.b + 1] - ln.pre[w.b], rem = x - before;
  w.g = rem / head;
  w.nb = line_blocks(ln, w.b);
  w.base = before + w.g * head;
  w.u = 0;
  if (ln.chunk != kNoChunks) {
    const unsigned ci = (x - w.base) / static_cast<unsigned>(ln.chunk + kUnitCost);
    w.u = ci * ln.chunk;
    w.base += ci * static_cast<unsigned>(ln.chunk + kUnitCost);
  }
  w.n = unit_blocks(ln, w.nb, w.u);
}
__device__ __forceinline__ void walk_start(const Line& ln, Walk& w, unsigned x, unsigned end, int lane) {
  w.end = end;
  w.more = false;
  w.b = w.g = w.u = w.n = w.nb = w.j = w.jend = 0;
  w.base = 0;
  if (x >= end) return;
  walk_unit(ln, w, x, lane);
  walk_range(w, x);
}
// the first place at or behind x where a unit begins
__device__ __forceinline__ unsigned next_unit(const Line& ln, unsigned x, int lane) {
  Walk w;
  walk_unit(ln, w, x, lane);
  return w.base == x ? x : w.base + w.n + kUnitCost;
}

// ---- warp-level pieces ------------------------------------------------------------------------------------------------
__device__ __forceinline__ void ldmatrix4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
__device__ __forceinline__ uint32_t transpose8x8(uint32_t x) {
  uint32_t y;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}
template <bool kE5m2> __device__ __forceinline__ uint32_t codes_lo(uint32_t w) { return kE5m2 ? e5m2x2_to_f16x2_lo(w) : e4m3x2_to_f16x2_lo(w); }
template <bool kE5m2> __device__ __forceinline__ uint32_t codes_hi(uint32_t w) { return kE5m2 ? e5m2x2_to_f16x2_hi(w) : e4m3x2_to_f16x2_hi(w); }

// Algorithm 1 phase 1 for one token, on the granule as it sits in shared memory (K part, V part, header), which is then
// written back: the write kernels' rule (write_part), with the same value for every number that is stored.
// k, v: this lane's D / 32 consecutive values of the token's rows, as packed pairs.
template <int D, bool kE5m2>
__device__ __noinline__ void append_token(uint8_t* st, uint8_t* gran, const uint2 k, const uint2 v, int off, int lane) {
  constexpr int kPart = kBlockSize * D, kPerLane = D / 32;
  float* hdr = reinterpret_cast<float*>(st + header_offset(D));
  const bool fresh = off == 0;
  const uint32_t raw[2][2] = {{k.x, k.y}, {v.x, v.y}};
  float s_old[2], s_new[2];
#pragma unroll
  for (int which = 0; which < 2; ++which) {
    uint32_t amax2 = raw[which][0] & 0x7FFF7FFFu;
    if (kPerLane == 4) amax2 = __vmaxu2(amax2, raw[which][1] & 0x7FFF7FFFu);
    const uint32_t am = __reduce_max_sync(0xffffffffu, max(amax2 << 16, amax2 & 0xFFFF0000u));   // non-negative floats order like their bits
    s_old[which] = fresh ? 0.0f : hdr[which];
    s_new[which] = fmaxf(s_old[which], __fdiv_rn(__uint_as_float(am), kE5m2 ? kE5m2Max : kE4m3Max));
  }
#pragma unroll
  for (int which = 0; which < 2; ++which) {
    uint8_t* part = st + which * kPart;
    if (fresh) {
      for (int i = lane; i < kPart / 16; i += 32) reinterpret_cast<uint4*>(part)[i] = make_uint4(0u, 0u, 0u, 0u);
    } else if (s_new[which] > s_old[which] && s_old[which] > 0.0f) {
#pragma unroll 4
      for (int i = lane; i < kPart; i += 32) {
        const float val = __fmul_rn(kE5m2 ? e5m2_to_f32(part[i]) : e4m3_to_f32(part[i]), s_old[which]);
        part[i] = static_cast<uint8_t>(kE5m2 ? f32_to_e5m2(__fdiv_rn(val, s_new[which])) : f32_to_e4m3(__fdiv_rn(val, s_new[which])));
      }
    }
  }
  __syncwarp();
#pragma unroll
  for (int which = 0; which < 2; ++which) {
#pragma unroll
    for (int e = 0; e < kPerLane; ++e) {
      const float x = (e & 1) ? bf16_hi(raw[which][e >> 1]) : bf16_lo(raw[which][e >> 1]);
      const float y = s_new[which] > 0.0f ? __fdiv_rn(x, s_new[which]) : x;
      st[which * kPart + (which == 0 ? k_elem_offset(D, true, off, lane * kPerLane + e) : v_elem_offset(D, true, off, lane * kPerLane + e))] =
          static_cast<uint8_t>(kE5m2 ? f32_to_e5m2(y) : f32_to_e4m3(y));
    }
  }
  if (lane < 8) hdr[lane] = lane == 0 ? s_new[0] : lane == 1 ? s_new[1] : fresh ? 0.0f : hdr[lane];
  __syncwarp();
  for (int i = lane; i < (2 * kPart + kFp8Header) / 16; i += 32) reinterpret_cast<uint4*>(gran)[i] = reinterpret_cast<const uint4*>(st)[i];
}
// This lane's D / 32 consecutive values of a row that may be aligned for no more than its elements.
template <int D>
__device__ __forceinline__ uint2 load_new(const __nv_bfloat16* row, bool vec, int lane) {
  uint32_t w[D / 64];
  if (vec) load_row<D / 32, true>(row + lane * (D / 32), w); else load_row<D / 32, false>(row + lane * (D / 32), w);
  return make_uint2(w[0], D == 128 ? w[D / 64 - 1] : 0u);
}

// A head's pieces merged by log-sum-exp: numerators of the lane's four dims, denominator, maximum.
struct Acc {
  float M, den;
  float4 num;
};
__device__ __forceinline__ void acc_clear(Acc& a) { a.M = -INFINITY; a.den = 0.0f; a.num = make_float4(0.0f, 0.0f, 0.0f, 0.0f); }
// Up to 32 more pieces into the accumulator.  Lane k brings piece k's maximum and sum; `rows(k)` is where the piece's o
// (normalised by its sum) lies for this lane.
template <bool kGlobal, class Rows>
__device__ __forceinline__ void acc_merge(Acc& a, int n, float m, float l, bool on, Rows rows) {
  constexpr int kUnroll = 4;
  float4 o[kUnroll];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int k = 0; k < kUnroll; ++k) {
      const float4* from = reinterpret_cast<const float4*>(rows(min(k0 + k, n - 1)));
      o[k] = on ? (kGlobal ? __ldcg(from) : *from) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
  };
  fetch(0);                              // (on their way while the weights are worked out)
  const bool some = l > 0.0f;
  const float top = fmaxf(a.M, ordered_to_f32(__reduce_max_sync(0xffffffffu, f32_to_ordered(some ? m : -INFINITY))));
  const float wgt = some ? l * ex2(m - top) : 0.0f;
  const float keep = a.den > 0.0f ? ex2(a.M - top) : 0.0f;
  a.num.x *= keep; a.num.y *= keep; a.num.z *= keep; a.num.w *= keep;
  a.den = a.den * keep + warp_sum(wgt);
  a.M = top;
#pragma unroll 1
  for (int k0 = 0;;) {
#pragma unroll
    for (int k = 0; k < kUnroll; ++k) {
      const float w = k0 + k < n ? __shfl_sync(0xffffffffu, wgt, k0 + k) : 0.0f;
      if (w > 0.0f) { a.num.x += w * o[k].x; a.num.y += w * o[k].y; a.num.z += w * o[k].z; a.num.w += w * o[k].w; }
    }
    k0 += kUnroll;
    if (k0 >= n) break;
    fetch(k0);
  }
}

// ---- units that several warps share: merged by log-sum-exp, one (unit, head) per warp at a time ---------------------------
// Pieces of the warps of a CTA lie in shared memory.  A head of a piece that other shares hold the rest of goes to the
// workspace, and is counted; who counts the last one takes them all and finishes the unit.  The first piece of a unit lies
// in the odd slot of its share, the others in the even ones.
template <int D, int FMT, int L>
struct Merge {
  using C = Cfg<D, FMT>;
  const DecodeParams& p;
  const LayerTable<L>& table;
  Line ln;
  uint8_t* smem;
  const Rec* recs;
  unsigned T;                            // places of a share
  int piece0_off, piece1_off;            // in a warp's part of shared memory
  int warp, lane, y;                     // y: the layer
  // What this warp has left in the workspace, lane i for the i-th piece: they are counted at once, so that the trips there
  // and back (about 1 us) are made side by side.
  int left = 0;
  int left_cta = 0, left_pieces = 0, left_b = 0, left_gh = 0, left_u = 0, left_region = 0;

  __device__ __forceinline__ bool on() const { return lane * 4 < D; }
  __device__ __forceinline__ size_t slot_of(int region, int cta, bool first, int h) const {
    return ((static_cast<size_t>(region) * p.shares + cta) * 2 + (first ? 1 : 0)) * p.group + h;
  }
  __device__ __forceinline__ void leave_piece(const Acc& a, int region, unsigned share, bool first, int b, int g, int h, int u, int cta_first, int pieces) {
    const size_t at = slot_of(region, share, first, h);
    const float dinv = a.den > 0.0f ? 1.0f / a.den : 0.0f;
    if (on()) *reinterpret_cast<float4*>(p.run_o + at * D + lane * 4) = make_float4(a.num.x * dinv, a.num.y * dinv, a.num.z * dinv, a.num.w * dinv);
    if (lane == 0) { p.run_m[at] = a.M; p.run_l[at] = a.den; }
    if (lane == left) { left_cta = cta_first; left_pieces = pieces; left_b = b; left_gh = g * p.group + h; left_u = u; left_region = region; }
    ++left;
  }
  __device__ __forceinline__ bool count_piece() const {      // one lane, behind the others' stores
    // release (this piece is visible before the count moves) and acquire (the other pieces are visible before they are read)
    int* counter = p.counters + (left_region * p.shares + left_cta) * kMaxGroup + left_gh % p.group;
    int old;
    asm volatile("atom.add.acq_rel.gpu.s32 %0, [%1], 1;" : "=r"(old) : "l"(counter) : "memory");
    if (old != left_pieces - 1) return false;
    *counter = 0;                        // ready for the next call
    return true;
  }
  __device__ __forceinline__ void take_pieces(Acc& a, int region, int cta_f, int pieces, int h) const {
    acc_clear(a);
#pragma unroll 1
    for (int c0 = 0; c0 < pieces; c0 += 32) {
      const int n = min(32, pieces - c0);
      auto slot = [&](int c) { return slot_of(region, cta_f + c, c == 0, h); };
      const float m = lane < n ? __ldcg(p.run_m + slot(c0 + lane)) : 0.0f, l = lane < n ? __ldcg(p.run_l + slot(c0 + lane)) : 0.0f;
      acc_merge<true>(a, n, m, l, on(), [&](int k) { return p.run_o + slot(c0 + k) * D + lane * 4; });
    }
  }
  __device__ __forceinline__ void store_out(const Acc& a, int b, int g, int h) const {
    const float dinv = a.den > 0.0f ? 1.0f / a.den : 0.0f;
    if (on()) *reinterpret_cast<uint2*>(table.l[L == 1 ? 0 : y].out + (static_cast<size_t>(b) * p.num_q_heads + g * p.group + h) * D + lane * 4) =
        make_uint2(pack_bf16x2(a.num.x * dinv, a.num.y * dinv), pack_bf16x2(a.num.z * dinv, a.num.w * dinv));
  }
  __device__ __forceinline__ void finish(const Acc& a, int b, int g, int h, int u) const {
    if (p.chunk_blocks == 0 || line_blocks(ln, b) <= ln.chunk) store_out(a, b, g, h);
    if (p.chunk_blocks > 0) {
      const size_t at = (static_cast<size_t>(b) * p.num_q_heads + g * p.group + h) * p.max_chunks + u / ln.chunk;
      const float dinv = a.den > 0.0f ? 1.0f / a.den : 0.0f;
      if (on()) *reinterpret_cast<float4*>(p.part_o + at * D + lane * 4) = make_float4(a.num.x * dinv, a.num.y * dinv, a.num.z * dinv, a.num.w * dinv);
      if (lane == 0) { p.part_m[at] = a.M * kLn2; p.part_l[at] = a.den * kUnshift; }
    }
  }
  // what the warps of this CTA hold of the units of a share
  __device__ __forceinline__ void local(unsigned share) {
    const int G = p.group;
    const int region = L > 1 ? y : p.chunk_blocks > 0 ? 1 : 0;
    const int flags = lane < C::kWarps ? recs[lane].flags : 0;
    const unsigned has0 = __ballot_sync(0xffffffffu, flags & kHas0), ends0 = __ballot_sync(0xffffffffu, flags & kEnds0), has1 = __ballot_sync(0xffffffffu, flags & kHas1);
    // a chain: the warps that hold pieces of one unit, the first of them `from` (kind 0: the unit began in another CTA)
    const int chains = static_cast<int>(has0 & 1u) + __popc(has1);
    static_assert((C::kWarps + 1) * kMaxGroup / C::kWarps + 3 <= 32, "a lane for every piece a warp leaves");
#pragma unroll 1
    for (int task = warp; task < chains * G; task += C::kWarps) {
      const int ci = task / G, h = task - ci * G;
      const int kind = (has0 & 1u) && ci == 0 ? 0 : 1;
      unsigned rest = has1;
      for (int k = static_cast<int>(has0 & 1u); k < ci; ++k) rest &= rest - 1;
      const int from = kind ? __ffs(rest) - 1 : 0;
      int last = from;
      bool closed = kind == 0 && (ends0 & 1u);
      if (!closed) {
        const int held = __ffs(~(has0 >> (from + 1))) - 1, end = __ffs(ends0 >> (from + 1));
        closed = end != 0 && end <= held;
        last = from + (closed ? end : held);
      }
      const int b = kind ? recs[from].b1 : recs[from].b0, g = kind ? recs[from].g1 : recs[from].g0, u = kind ? recs[from].u1 : recs[from].u0;
      auto piece = [&](int k) {
        return reinterpret_cast<const float*>(smem + (from + k) * C::kWarpBytes + ((kind && k == 0) ? piece1_off : piece0_off)) + h * C::kPieceStride;
      };
      const int n = last - from + 1;
      Acc a;
      acc_clear(a);
      acc_merge<false>(a, n, lane < n ? piece(lane)[D] : 0.0f, lane < n ? piece(lane)[D + 1] : 0.0f, on(), [&](int k) { return piece(k) + lane * 4; });
      if (kind && closed) {
        finish(a, b, g, h, u);
      } else {
        const unsigned first = unit_place(ln, b, g, u) + kUnitCost;
        const int nu = unit_blocks(ln, line_blocks(ln, b), u), cta_f = first / T;
        leave_piece(a, region, share, kind != 0, b, g, h, u, cta_f, static_cast<int>((first + nu - 1) / T) - cta_f + 1);
      }
    }
  }
  // the pieces left in the workspace: counted, and units finished of which they were the last.  (In chunk mode region 0 has
  // whole (sequence, kv head) pairs, of which the output is due, region 1 chunks.)
  __device__ __forceinline__ void count_and_finish() const {
    __syncwarp();
    unsigned last = __ballot_sync(0xffffffffu, left_pieces > 0 && count_piece());
    __syncwarp();                        // the others' pieces, which a lane has acquired, are there for all lanes
#pragma unroll 1
    for (; last != 0; last &= last - 1) {
      const int i = __ffs(last) - 1, gh = __shfl_sync(0xffffffffu, left_gh, i), g = gh / p.group, h = gh - g * p.group;
      const int region = __shfl_sync(0xffffffffu, left_region, i), b = __shfl_sync(0xffffffffu, left_b, i), u = __shfl_sync(0xffffffffu, left_u, i);
      Acc a;
      take_pieces(a, region, __shfl_sync(0xffffffffu, left_cta, i), __shfl_sync(0xffffffffu, left_pieces, i), h);
      if (L == 1 && p.chunk_blocks > 0 && region == 0) store_out(a, b, g, h); else finish(a, b, g, h, u);
    }
  }
};

template <int D, int FMT, int L>
__global__ void __launch_bounds__(Cfg<D, FMT>::kThreads, kCtasPerSm) paged_decode_kernel(const __grid_constant__ DecodeParams p, const __grid_constant__ LayerTable<L> table) {
  using C = Cfg<D, FMT>;
  constexpr int kQSteps = D / 16;
  extern __shared__ __align__(128) uint8_t smem[];
  int* lens = reinterpret_cast<int*>(smem + C::kLensOff);
  unsigned* pre = reinterpret_cast<unsigned*>(smem + C::kPreOff);
  Rec* recs = reinterpret_cast<Rec*>(smem + C::kRecOff);
  int* misc = reinterpret_cast<int*>(smem + C::kMiscOff);   // [0..15] warps' sums, [16] wrong plan, [17..32] warps' longest unit
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int row = lane >> 2, quad = lane & 3;
  const int B = p.batch, Hkv = p.num_kv_heads, G = p.group, Hq = p.num_q_heads;
  uint8_t* ring = smem + warp * C::kWarpBytes;
  constexpr int piece0_off = C::kStages * C::kGran;
  const int piece1_off = L == 1 ? 0 : piece0_off + G * C::kPieceStride * 4;                        // in a warp's shared memory
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::kBarOff) + warp * C::kStages;
  uint64_t* bar_pieces = reinterpret_cast<uint64_t*>(smem + C::kBarOff) + C::kWarps * C::kStages;   // every warp has left its pieces
  uint64_t* bar_merged = bar_pieces + 1;                                                            // .. has no more use for the others' pieces

  COOPT_TRACE_CYCLES(p.trace, kTrEntry, tid == 0);
#ifdef COOPT_TRACE
  if (tid == 0 && p.trace != nullptr && blockIdx.x < kTraceMaxCtas) {
    trace_put(p.trace, kTrPrevExitNs, p.trace[blockIdx.x * kTraceSlots + kTrExitNs]);
    unsigned int smid;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
    trace_put(p.trace, kTrSmId, smid + 1);
  }
#endif
  COOPT_TRACE_NS(p.trace, kTrEntryNs, tid == 0);
  if (lane == 0) {
    for (int i = 0; i < C::kStages; ++i) mbar_init(&bars[i], 1);
    if (warp == 0) { mbar_init(bar_pieces, C::kWarps); mbar_init(bar_merged, C::kWarps); }
    mbar_fence_init();
  }
  const auto layer = [&](int y) -> const LayerPtrs& { return table.l[L == 1 ? 0 : y]; };
  // Launched as a programmatic dependent, this CTA may run while the kernel before it still does; p.order says what
  // may be read before that one has finished.  (The kernel behind this one may start only then, too: it may read early
  // what the kernel before this one wrote.)
  if (p.order == kDependent) wait_previous_kernel();

  // ---- the line: context lengths and their prefix sums -------------------------------------------------------
  {
    constexpr int kPer = (kMaxBatch + C::kThreads - 1) / C::kThreads;
    const int chunk = p.chunk_blocks > 0 ? p.chunk_blocks : kNoChunks;
    unsigned v[kPer], sum = 0;
    int most = 0, key = p.plan_key;
    bool empty = false;
    if (tid == 0 && p.plan != nullptr) key = p.plan->key;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int b = tid * kPer + k;
      int len = b < B ? p.context_lens[b] : 0;
      len = max(0, min(len, p.max_blocks_per_seq * kBlockSize));
      if (b < B) lens[b] = len;
      const int nb = (len + kBlockSize - 1) / kBlockSize;
      const int units = nb == 0 ? 0 : (chunk == kNoChunks ? 1 : (nb + chunk - 1) / chunk);
      v[k] = nb + units * kUnitCost;
      sum += v[k];
      most = max(most, min(nb, chunk));
      empty = empty || (b < B && nb == 0);
    }
    most = __reduce_max_sync(0xffffffffu, most) + (__any_sync(0xffffffffu, empty) ? kSomeEmpty : 0);
    unsigned inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    if (lane == 31) { misc[warp] = inc; misc[17 + warp] = most; }
    if (tid == 0) misc[16] = key != p.plan_key;
    __syncthreads();
    unsigned at = inc - sum;
    for (int w = 0; w < warp; ++w) at += misc[w];
    if (tid == 0) pre[0] = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      at += v[k];
      if (tid * kPer + k < B) pre[tid * kPer + k + 1] = at;
    }
    __syncthreads();
  }
  if (misc[16]) {                                  // not a plan of this problem (uniform over the grid)
    if (p.order != kDependent) wait_previous_kernel();
    if (tid == 0) atomicCAS(p.status, 0, COOPT_ERR_INVALID_ARG);
    return;
  }
  COOPT_TRACE_CYCLES(p.trace, kTrLine, tid == 0);
  Line ln;
  ln.lens = lens; ln.pre = pre; ln.batch = B; ln.heads = Hkv; ln.chunk = p.chunk_blocks > 0 ? p.chunk_blocks : kNoChunks;
  // A share: T places of a layer's line.  A layer is cut the same way whatever else the launch does, so its result does
  // not depend on how many layers share the launch.  CTA i takes the shares i, i + grid, .. of all layers, one layer
  // behind the other; the copies of a share are under way while the pieces of the one before are merged.
  const unsigned places = Hkv * pre[B];
  unsigned T = max(static_cast<unsigned>(kMinPlaces), (places + p.shares - 1) / p.shares);
  // Shared units cost a trip through the workspace at the end of a share.  Where units are short, a share holds the units
  // that begin among its places whole instead.  (In chunk mode every share between the first and the last of a (sequence,
  // kv head) has to hold a chunk of it.)
  int most = 0;
  bool none_empty = true;
  for (int k = 0; k < C::kWarps; ++k) {
    const int m = misc[17 + k];
    none_empty = none_empty && m < kSomeEmpty;
    most = max(most, m & (kSomeEmpty - 1));
  }
  const bool whole = most * (D / 64) <= (T == kMinPlaces ? C::kWholeIdle : kWholeUnits) && (p.chunk_blocks == 0 || most + kUnitCost <= static_cast<int>(T));
  // Where they are very short, a warp holds whole what begins among its places, and nothing is merged.  Nor does a unit's
  // result depend on the shares then: they are made as large as it takes for every CTA to have one at most.
  const bool solo = whole && p.chunk_blocks == 0 && most <= p.solo_blocks;
  if (L > 1 && solo) {
    const unsigned m = max(1u, gridDim.x / p.layers);
    T = max(T, (places + m - 1) / m);
  }
  // Where a layer does not fill the device, its shares are its units: as many at a time as there are CTAs, of whichever layer.
  // (Three layers of 17 sequences of 854 tokens, two kv heads: 35.4 us with shares of 16 places, most of them empty and the
  // others unevenly spread over the CTAs, 14.1 so; eight of 7 sequences of 272..544 tokens, four kv heads: 29.7 / 20.5.)
  const bool by_unit = whole && !solo && p.chunk_blocks == 0 && T == kMinPlaces && none_empty && B * Hkv <= p.shares;
  const unsigned shares = by_unit ? B * Hkv : (places + T - 1) / T, all_shares = L == 1 ? shares : shares * p.layers;
  // What is looked at seldom waits in shared memory, a copy for every warp, and not in registers that the loop over blocks
  // needs: the walk of the copies (once in 32 blocks), its share, and how shares are cut.
  Walk* copy_walk = reinterpret_cast<Walk*>(smem + C::kCopyWalkOff + warp * 128);
  Walk* work_walk = copy_walk + 1;
  unsigned* copy_share = reinterpret_cast<unsigned*>(copy_walk) + 24;
  volatile unsigned* cut = copy_share + 1;                              // [0] bit 0: whole, bit 1: solo, bit 2: by unit; [1] T
  if (lane == 0) { cut[0] = by_unit ? 4u : (whole ? 1u : 0u) | (solo ? 2u : 0u); cut[1] = T; }
  __syncwarp();
  auto share_range = [&](unsigned v, unsigned& lo, unsigned& hi) {       // places of a layer's share v
    lo = v * T;
    hi = min(places, lo + T);
    if (whole) {
      lo = next_unit(ln, lo, lane);
      hi = hi < places ? next_unit(ln, hi, lane) : places;
    }
  };
  auto share_layer = [&](unsigned s) -> int { return L == 1 ? 0 : s / shares; };
  auto share_walk = [&](unsigned s, Walk& w) {                          // this warp's part of share s
    // (Three look-ups at most, in a loop: code that a CTA runs once is bound by the fetch of its instructions.)
    const unsigned T = cut[1], mode = cut[0];
    const bool solo = (mode & 2u) != 0;
    const unsigned v = L == 1 ? s : s % shares;
    unsigned lo = v * T, hi = min(places, lo + T), x = lo;
    w.more = false;
    if ((mode & 4u) != 0) {
      const unsigned b = v / Hkv, head = pre[b + 1] - pre[b];
      lo = Hkv * pre[b] + (v - b * Hkv) * head;
      hi = lo + head;
    }
    if (solo) {
      const unsigned Tw = (T + C::kWarps - 1) / C::kWarps;
      x = min(hi, lo + warp * Tw);
      hi = min(hi, x + Tw);
    }
#pragma unroll 1
    for (int step = (mode & 1u) != 0 ? 0 : 2; step < 3; ++step) {
      if (step == 1) x = hi;
      if (step == 2) {
        const unsigned mine = hi > lo ? hi - lo : 0u, Tw = (mine + C::kWarps - 1) / C::kWarps;
        x = solo ? lo : min(hi, lo + warp * Tw);
        w.end = solo ? hi : min(hi, x + Tw);
        if (x >= w.end) return;
      }
      if (x < places) walk_unit(ln, w, x, lane);
      const unsigned next = x >= places || w.base == x ? x : w.base + w.n + kUnitCost;
      if (step == 0) lo = next;
      if (step == 1) hi = next;
    }
    walk_range(w, x);
  };
  // this warp's first unit in share s or, over several layers, in a later one (s moves there); and its next one
  auto walk_later = [&](unsigned& s, Walk& w) {
    if constexpr (L > 1) {
      while (!w.more && s + gridDim.x < all_shares) {
        s += gridDim.x;
        share_walk(s, w);
      }
    }
  };
  auto walk_on = [&](unsigned& s, Walk& w) {
    walk_next(ln, w);
    walk_later(s, w);
  };

  // ---- copies: a granule per request, a ring of stages per warp -------------------------------------------------
  // Physical block ids are looked up 32 at a time (one per lane), one batch ahead of the copies that need them.
  Walk w;                                          // where this warp's work is (in share `share`), and where its copies are (in share `ps`)
  unsigned ps = blockIdx.x;
  w.more = false;
  if (ps < all_shares) share_walk(ps, w);
  Walk fw = w;
  if (ps < all_shares) walk_later(ps, fw);                              // the first unit, and its layer
  const int fy = share_layer(ps);
  int ids_a = 0, g_a = 0, y_a = 0;
  int cnt_a = 0, pos_a = 0, ids_b = 0, cnt_b = 0, g_b = 0, y_b = 0;
  auto prefetch_q = [&](int y, int b, int g) {
    if (lane < G * D / 64) prefetch_l2(reinterpret_cast<const uint8_t*>(layer(y).q + (static_cast<size_t>(b) * Hq + g * G) * D) + lane * 128);
  };
  auto fetch_ids = [&]() {
    Walk pw = *copy_walk;
    unsigned ps = *copy_share;
    cnt_b = 0;
    if (!pw.more) return;
    cnt_b = min(32, pw.jend - pw.j);
    g_b = pw.g;
    y_b = share_layer(ps);
    ids_b = lane < cnt_b ? p.block_table[static_cast<size_t>(pw.b) * p.max_blocks_per_seq + pw.u + pw.j + lane] : 0;
    pw.j += cnt_b;
    if (pw.j >= pw.jend) {
      walk_on(ps, pw);
      if (pw.more) prefetch_q(share_layer(ps), pw.b, pw.g);
    }
    __syncwarp();
    if (lane == 0) { *copy_walk = pw; *copy_share = ps; }
    __syncwarp();
  };
  auto take_ids = [&]() {
    int id = ids_b;
    if (id < 0 || id >= p.num_blocks) {            // reported, and replaced by block 0: never dereferenced
      if (p.plan == nullptr) atomicCAS(p.status, 0, COOPT_ERR_INVALID_ARG);
      id = 0;
    }
    ids_a = id; g_a = g_b; y_a = y_b;
    cnt_a = cnt_b; pos_a = 0;
    fetch_ids();
  };
  uint32_t issued = 0, consumed = 0;               // copies, and the stages that take the next one and hold the oldest one
  int in_stage = 0, out_stage = 0;
  uint32_t out_phase = 0;
  auto issue = [&]() {
    if (pos_a == cnt_a) take_ids();
    if (pos_a < cnt_a) {
      const int id = __shfl_sync(0xffffffffu, ids_a, pos_a);
      ++pos_a;
      const int stage = in_stage;
      if (++in_stage == C::kStages) in_stage = 0;
      if (lane == 0) {
        mbar_expect_tx(&bars[stage], C::kCopy);
        bulk_copy_g2s(ring + stage * C::kGran, layer(y_a).cache + (static_cast<size_t>(id) * Hkv + g_a) * C::kGran, C::kCopy, &bars[stage]);
      }
      ++issued;
    }
  };

  // ---- per-lane constants of the operand layouts ---------------------------------------------------------------
  // FP8: ldmatrix row i of the "low" matrix of a K chunk is token 4 (i / 2) + i % 2, of the "high" one that token + 2
  const int kt = 4 * ((lane & 7) >> 1) + (lane & 1) + 2 * ((lane >> 3) & 1);
  const uint32_t k_lane = (kt >> 3) * 8 * D + (lane >> 4) * 128 + (kt & 7) * 16;
  const int tok0 = C::kFp8 ? 4 * (row >> 1) + (row & 1) : row;       // token of this lane's logits 0 and 1; 2 and 3: tok0 + kTokStep
  constexpr int kTokStep = C::kFp8 ? 2 : 8;

  // raw query rows: this lane's head is `row`, its dims as the contraction takes them.  (The first unit's are requested ahead of
  // its blocks; those of later units come from L2, where they have been requested with the unit's first block ids: registers
  // that hold them through the unit before cost more than the trip.)
  uint32_t qraw[kQSteps][2];
  auto load_q = [&](int y, int b, int g) {
    const bool live = row < G;
    const __nv_bfloat16* qp = layer(y).q + (static_cast<size_t>(b) * Hq + g * G + (live ? row : 0)) * D;
#pragma unroll
    for (int s = 0; s < kQSteps; ++s) {
      if constexpr (C::kFp8) {
        const uint2 v = live ? *reinterpret_cast<const uint2*>(qp + 16 * s + 4 * quad) : make_uint2(0u, 0u);
        qraw[s][0] = v.x; qraw[s][1] = v.y;
      } else {
        qraw[s][0] = live ? *reinterpret_cast<const uint32_t*>(qp + 16 * s + 2 * quad) : 0u;
        qraw[s][1] = live ? *reinterpret_cast<const uint32_t*>(qp + 16 * s + 2 * quad + 8) : 0u;
      }
    }
  };
  bool dead = false;
  // What the first unit needs besides its blocks is on its way to L2 before the copies queue up in front of it (also where
  // the kernel before may still write it: L2 is where its stores arrive).
  if (fw.more) {
    const LayerPtrs& io = layer(fy);
    prefetch_q(fy, fw.b, fw.g);
    if (io.k_new != nullptr && lane < 3) {
      const long long at = static_cast<long long>(fw.b) * p.kv_token_stride + fw.g * D;
      prefetch_l2(lane == 0 ? static_cast<const void*>(io.k_new + at) : lane == 1 ? static_cast<const void*>(io.v_new + at) : static_cast<const void*>(io.slot_mapping + fw.b));
    }
  }
  if (lane == 0) { *copy_walk = fw; *copy_share = ps; }
  __syncwarp();
  fetch_ids();
#pragma unroll 1
  for (int step = 0; step < 2; ++step) {
    if ((step == 0) == (p.order == kOverlapPrevious)) {
#pragma unroll 1
      for (int i = 0; i < C::kStages; ++i) issue();
      COOPT_TRACE_CYCLES(p.trace, kTrFirstCopy, tid == 0);
    } else {
      if (p.order != kDependent) wait_previous_kernel();
      COOPT_TRACE_CYCLES(p.trace, kTrPrevDone, tid == 0);
      if (fw.more) load_q(fy, fw.b, fw.g);
    }
  }
  if (blockIdx.x == 0) {
    if (p.plan != nullptr && tid < kPlanCtas && p.plan->status[tid] != 0) atomicCAS(p.status, 0, p.plan->status[tid]);
    // coopt_paged_chunked takes this path only for one query token per sequence: any other split of the same total is reported
    if (p.cu_q_lens != nullptr)
      for (int b = tid; b <= B; b += C::kThreads)
        if (p.cu_q_lens[b] != b) atomicCAS(p.status, 0, COOPT_ERR_INVALID_ARG);
  }
  // sequences with an empty context: all-zero output rows
  for (int b = blockIdx.x; b < B; b += gridDim.x)
    if (lens[b] == 0)
      for (int y = 0; y < (L == 1 ? 1 : p.layers); ++y)
        for (int i = tid; i < Hq * D / 8; i += C::kThreads) reinterpret_cast<uint4*>(layer(y).out + static_cast<size_t>(b) * Hq * D)[i] = make_uint4(0u, 0u, 0u, 0u);

  uint32_t round = 0;
#pragma unroll 1
  for (unsigned share = blockIdx.x; share < all_shares; share += gridDim.x, ++round) {
  const int y = share_layer(share);
  const unsigned v_share = L == 1 ? share : share - y * shares;
  if (round > 0) share_walk(share, w);
  int flags = 0;                         // of the pieces this warp leaves (Rec)
#pragma unroll 1
  while (w.more) {
    if (consumed != 0) load_q(y, w.b, w.g);
    // ---- query operand: f16 (exact: rows scaled by a power of two), or bf16 as it is -------------------------------
    uint32_t qf[kQSteps][2];
    float qs[2];                                   // logit scale of heads 2 quad, 2 quad + 1
    if constexpr (C::kFp8) {
      uint32_t amax2 = 0;
#pragma unroll
      for (int s = 0; s < kQSteps; ++s) amax2 = __vmaxu2(__vmaxu2(amax2, qraw[s][0] & 0x7FFF7FFFu), qraw[s][1] & 0x7FFF7FFFu);
      uint32_t am = max(amax2 << 16, amax2 & 0xFFFF0000u);
      am = max(am, __shfl_xor_sync(0xffffffffu, am, 1));
      am = max(am, __shfl_xor_sync(0xffffffffu, am, 2));
      int k2 = 0;
      if (am != 0u) k2 = max(-64, min(64, 134 - static_cast<int>((am >> 23) & 0xFF)));
      const float up = __uint_as_float(static_cast<uint32_t>(k2 + 127) << 23);
      const float down = p.sm_scale_log2 * __uint_as_float(static_cast<uint32_t>(127 - k2) << 23);
#pragma unroll
      for (int s = 0; s < kQSteps; ++s)
#pragma unroll
        for (int e = 0; e < 2; ++e) qf[s][e] = pack_f16x2(bf16_lo(qraw[s][e]) * up, bf16_hi(qraw[s][e]) * up);
      qs[0] = __shfl_sync(0xffffffffu, down, 8 * quad);
      qs[1] = __shfl_sync(0xffffffffu, down, 8 * quad + 4);
    } else {
#pragma unroll
      for (int s = 0; s < kQSteps; ++s) { qf[s][0] = qraw[s][0]; qf[s][1] = qraw[s][1]; }
      qs[0] = qs[1] = p.sm_scale_log2;
    }
    COOPT_TRACE_CYCLES(p.trace, kTrQuery, tid == 0 && consumed == 0 && qf[0][0] != 0x12345u);
    float o[D / 16][4];
#pragma unroll
    for (int t = 0; t < D / 16; ++t)
#pragma unroll
      for (int e = 0; e < 4; ++e) o[t][e] = 0.0f;
    float m[2] = {-INFINITY, -INFINITY}, top[2] = {-INFINITY, -INFINITY}, l[2] = {0.0f, 0.0f};
    float vref = 0.0f, vinv = 0.0f;
    // what the loop over blocks needs of the walk; the rest waits in shared memory
    const int j_end = w.jend, valid = lens[w.b] - w.u * kBlockSize;            // (the end of the context, counted from the unit's start)
    if (lane == 0) *work_walk = w;
    __syncwarp();

#pragma unroll 1
    for (int j = w.j; j < j_end && !dead; ++j) {
      // (The one test that every block meets: whether it is the last of the context.)
      const bool last = (j + 1) * kBlockSize >= valid;
      int seen = kBlockSize;                                                 // tokens of the block (Eq. 9)
      // the step's new token: what it needs is loaded while its block is on the way
      bool append = false;
      long long slot = -1;
      int id = 0;
      uint2 k_row = make_uint2(0u, 0u), v_row = k_row;
      if (last) {
        seen = valid - j * kBlockSize;
        if constexpr (C::kFp8) {
          append = layer(y).k_new != nullptr;
          if (append) {
            const LayerPtrs& io = layer(y);
            const bool vec = ((reinterpret_cast<uintptr_t>(io.k_new) | reinterpret_cast<uintptr_t>(io.v_new) | static_cast<uintptr_t>(p.kv_token_stride * 2)) & (D / 16 - 1)) == 0;
            const long long at = static_cast<long long>(work_walk->b) * p.kv_token_stride + work_walk->g * D;
            slot = io.slot_mapping[work_walk->b];
            id = p.block_table[static_cast<size_t>(work_walk->b) * p.max_blocks_per_seq + work_walk->u + j];
            k_row = load_new<D>(io.k_new + at, vec, lane);
            v_row = load_new<D>(io.v_new + at, vec, lane);
          }
        }
      }
      // the oldest copy in flight (the next one's place is worked out while this one is waited for: eight layers of 64 x 100..5000
      // tokens, head_dim 64, 180.5 us behind the wait, 173.4 so)
      uint8_t* const st = ring + out_stage * C::kGran;
      const bool there = mbar_wait_bounded(&bars[out_stage], out_phase);
      if (++out_stage == C::kStages) { out_stage = 0; out_phase ^= 1u; }
      dead = !__all_sync(0xffffffffu, there);
      COOPT_TRACE_CYCLES(p.trace, kTrFirstLanded, tid == 0 && consumed == 0);
      if (dead) {                                  // (the stage that was waited for stays the oldest)
        if (--out_stage < 0) { out_stage += C::kStages; out_phase ^= 1u; }
        break;
      }
      ++consumed;
      if constexpr (C::kFp8) {
        if (last) {
          if (append && slot >= 0) {                                         // Eq. 5: negative slots are skipped
            const int off = (valid - 1) % kBlockSize;
            if (slot != static_cast<long long>(id) * kBlockSize + off) {     // not the sequence's last position
              if (lane == 0) atomicCAS(p.status, 0, COOPT_ERR_INVALID_ARG);
            } else if (id >= 0 && id < p.num_blocks) {
              append_token<D, C::kE5m2>(st, layer(y).cache + (static_cast<size_t>(id) * Hkv + work_walk->g) * C::kGran, k_row, v_row, off, lane);
            }
            __syncwarp();
          }
          if (seen < kBlockSize) {                 // V codes of slots past the context are cleared: they may hold anything
            auto mask = [&](int word) { return seen >= 4 * word + 4 ? 0xFFFFFFFFu : seen <= 4 * word ? 0u : (1u << (8 * (seen - 4 * word))) - 1u; };
#pragma unroll
            for (int i = 0; i < D / 32; ++i) {
              uint4* row = reinterpret_cast<uint4*>(st + kBlockSize * D) + i * 32 + lane;        // 16 tokens of a dim
              const uint4 v = *row;
              *row = make_uint4(v.x & mask(0), v.y & mask(1), v.z & mask(2), v.w & mask(3));
            }
            __syncwarp();
          }
        }
      }

      // ---- S^T = K Q^T: 16 tokens x 8 heads ------------------------------------------------------------------------
      float sa[4] = {0.0f, 0.0f, 0.0f, 0.0f}, sb[4] = {0.0f, 0.0f, 0.0f, 0.0f};
      float sk = 1.0f, sv = 1.0f;
      if constexpr (C::kFp8) {
        const float2 hdr = *reinterpret_cast<const float2*>(st + header_offset(D));
        sk = hdr.x; sv = hdr.y;
#pragma unroll
        for (int c = 0; c < D / 32; ++c) {
          uint32_t r[4];
          ldmatrix4(smem_u32(st) + k_lane + c * 256, r);
          mma16816<true>(sa, codes_lo<C::kE5m2>(r[0]), codes_lo<C::kE5m2>(r[1]), codes_hi<C::kE5m2>(r[0]), codes_hi<C::kE5m2>(r[1]), qf[2 * c][0], qf[2 * c][1]);
          mma16816<true>(sb, codes_lo<C::kE5m2>(r[2]), codes_lo<C::kE5m2>(r[3]), codes_hi<C::kE5m2>(r[2]), codes_hi<C::kE5m2>(r[3]), qf[2 * c + 1][0], qf[2 * c + 1][1]);
        }
      } else {
        const uint8_t* kp = st + lane * 16;
#pragma unroll
        for (int i = 0; i < D / 32; ++i) {
          const uint4 w0 = lds128(kp + i * 512), w1 = lds128(kp + (D / 32 + i) * 512);
          mma16816<false>(sa, w0.x, w1.x, w0.y, w1.y, qf[2 * i][0], qf[2 * i][1]);
          mma16816<false>(sb, w0.z, w1.z, w0.w, w1.w, qf[2 * i + 1][0], qf[2 * i + 1][1]);
        }
      }

      // ---- online softmax (Eq. 10) in base-2 units; the reference maximum is lazy --------------------------------------
      // (Each block goes by the references that it finds or moves itself.  Two blocks by one: far below what the second moves, the
      // first one's probabilities are f16 numbers of few bits, or zero.)
      const float k0 = qs[0] * sk, k1 = qs[1] * sk;
      float x[4] = {(sa[0] + sb[0]) * k0, (sa[1] + sb[1]) * k1, (sa[2] + sb[2]) * k0, (sa[3] + sb[3]) * k1};
      if (seen < kBlockSize) {
        if (tok0 >= seen) x[0] = x[1] = -INFINITY;
        if (tok0 + kTokStep >= seen) x[2] = x[3] = -INFINITY;
      }
      const float t0 = fmaxf(x[0], x[2]), t1 = fmaxf(x[1], x[3]);
      if constexpr (L == 1) {                      // (for exported partials)
        top[0] = fmaxf(top[0], t0);
        top[1] = fmaxf(top[1], t1);
      }
      const bool grow = C::kFp8 && sv > vref;
      if (__any_sync(0xffffffffu, t0 > m[0] + kLag || t1 > m[1] + kLag) || grow) {
        float f[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float t = h ? t1 : t0;
          t = fmaxf(t, __shfl_xor_sync(0xffffffffu, t, 4));
          t = fmaxf(t, __shfl_xor_sync(0xffffffffu, t, 8));
          t = fmaxf(t, __shfl_xor_sync(0xffffffffu, t, 16));
          const float mn = fmaxf(m[h], t);
          f[h] = ex2(m[h] - mn);
          m[h] = mn;
          l[h] *= f[h];
        }
        if (grow) {                                // (a reference is a normal number: its reciprocal is one then, too)
          const float vnew = fmaxf(sv, FLT_MIN);
          vinv = 1.0f / vnew;
          const float fv = vref * vinv;
          f[0] *= fv; f[1] *= fv;
          vref = vnew;
        }
#pragma unroll
        for (int t = 0; t < D / 16; ++t) { o[t][0] *= f[0]; o[t][1] *= f[1]; o[t][2] *= f[0]; o[t][3] *= f[1]; }
      }
      const float b0 = kShift - m[0], b1 = kShift - m[1];
      float pr[4];
      pr[0] = ex2(x[0] + b0); pr[1] = ex2(x[1] + b1); pr[2] = ex2(x[2] + b0); pr[3] = ex2(x[3] + b1);
      l[0] += pr[0] + pr[2];
      l[1] += pr[1] + pr[3];

      // ---- O^T += V^T P^T -----------------------------------------------------------------------------------------------
      if constexpr (C::kFp8) {
        const float pv = sv * vinv;
        const uint32_t p0 = transpose8x8(pack_f16x2(pr[0] * pv, pr[1] * pv)), p1 = transpose8x8(pack_f16x2(pr[2] * pv, pr[3] * pv));
#pragma unroll
        for (int c = 0; c < D / 32; ++c) {
          uint32_t r[4];
          ldmatrix4(smem_u32(st) + kBlockSize * D + lane * 16 + c * 512, r);
          mma16816<true>(o[2 * c], codes_lo<C::kE5m2>(r[0]), codes_lo<C::kE5m2>(r[1]), codes_hi<C::kE5m2>(r[0]), codes_hi<C::kE5m2>(r[1]), p0, p1);
          mma16816<true>(o[2 * c + 1], codes_lo<C::kE5m2>(r[2]), codes_lo<C::kE5m2>(r[3]), codes_hi<C::kE5m2>(r[2]), codes_hi<C::kE5m2>(r[3]), p0, p1);
        }
      } else {
        // bf16 probabilities as a high and a low half (16 bits in all)
        const uint32_t h0 = pack_bf16x2(pr[0], pr[1]), h1 = pack_bf16x2(pr[2], pr[3]);
        const uint32_t e0 = pack_bf16x2(pr[0] - bf16_lo(h0), pr[1] - bf16_hi(h0)), e1 = pack_bf16x2(pr[2] - bf16_lo(h1), pr[3] - bf16_hi(h1));
        const uint32_t p0 = transpose8x8(h0), p1 = transpose8x8(h1), r0 = transpose8x8(e0), r1 = transpose8x8(e1);
        const uint8_t* vp = st + part_offset(D, false, 1) + lane * 16;
        uint32_t m0 = 0xFFFFFFFFu, m1 = 0xFFFFFFFFu;
        if (seen < kBlockSize) {
          m0 = (2 * quad < seen ? 0x0000FFFFu : 0u) | (2 * quad + 1 < seen ? 0xFFFF0000u : 0u);
          m1 = (2 * quad + 8 < seen ? 0x0000FFFFu : 0u) | (2 * quad + 9 < seen ? 0xFFFF0000u : 0u);
        }
#pragma unroll
        for (int i = 0; i < D / 16; ++i) {
          const uint4 v = lds128(vp + i * 512);
          mma16816<false>(o[i], v.x & m0, v.z & m0, v.y & m1, v.w & m1, p0, p1);
          mma16816<false>(o[i], v.x & m0, v.z & m0, v.y & m1, v.w & m1, r0, r1);
        }
      }

      // ---- the stage goes back to the copy engine ---------------------------------------------------------------------
      __syncwarp();
      if (lane == 0) fence_proxy_async();
      issue();
    }
    w = *work_walk;
    __syncwarp();
    // ---- end of the unit (or of this warp's piece of it) ----------------------------------------------------------------
    if constexpr (C::kFp8) {
      if (__builtin_expect(vref < 0x1p-64f && vref > 0.0f, 0)) {      // (vref / l would lose bits among the subnormals)
#pragma unroll
        for (int t = 0; t < D / 16; ++t)
#pragma unroll
          for (int e = 0; e < 4; ++e) o[t][e] *= 0x1p-64f;
        vref *= 0x1p64f;
      }
    }
    float inv[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
      for (int s = 4; s <= 16; s <<= 1) l[h] += __shfl_xor_sync(0xffffffffu, l[h], s);
      inv[h] = l[h] > 0.0f ? (C::kFp8 ? vref : 1.0f) / l[h] : 0.0f;      // o and l go by the same reference
      if (L == 1 && p.chunk_blocks > 0) {          // exported partials carry the true maximum
#pragma unroll
        for (int s = 4; s <= 16; s <<= 1) top[h] = fmaxf(top[h], __shfl_xor_sync(0xffffffffu, top[h], s));
        l[h] *= ex2(m[h] - top[h]);
        m[h] = top[h];
      }
    }
    const bool starts = w.j == 0, ends = w.jend == w.n;
    if (starts && ends && w.n == w.nb) {
      // the whole (sequence, kv head): bf16 rows, transposed so that a lane holds pairs of dims of head `row`
      __nv_bfloat16* dst = layer(y).out + (static_cast<size_t>(w.b) * Hq + w.g * G + row) * D + 2 * quad;
#pragma unroll
      for (int t = 0; t < D / 16; ++t) {
        const uint32_t a = transpose8x8(pack_bf16x2(o[t][0] * inv[0], o[t][1] * inv[1])), c = transpose8x8(pack_bf16x2(o[t][2] * inv[0], o[t][3] * inv[1]));
        if (row < G) {
          *reinterpret_cast<uint32_t*>(dst + 16 * t) = a;
          *reinterpret_cast<uint32_t*>(dst + 16 * t + 8) = c;
        }
      }
    }
    if (starts && ends && p.chunk_blocks > 0) {
      // a whole chunk: exported
      const size_t rows = static_cast<size_t>(p.max_chunks);
      const size_t at = (static_cast<size_t>(w.b) * Hq + w.g * G + 2 * quad) * rows + w.u / ln.chunk;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (2 * quad + h < G) {
          float* dst = p.part_o + (at + h * rows) * D + row;
#pragma unroll
          for (int t = 0; t < D / 16; ++t) { dst[16 * t] = o[t][h] * inv[h]; dst[16 * t + 8] = o[t][2 + h] * inv[h]; }
          if (row == 0) { p.part_m[at + h * rows] = m[h] * kLn2; p.part_l[at + h * rows] = l[h] * kUnshift; }
        }
      }
    }
    if (!(starts && ends)) {
      // a piece: into shared memory, once the pieces of the share before are of no more use
      if (L > 1 && round > 0 && flags == 0 && !dead) dead = !__all_sync(0xffffffffu, mbar_wait_bounded(bar_merged, (round - 1) & 1u));
      float* piece = reinterpret_cast<float*>(ring + (starts ? piece1_off : piece0_off));
      float* at = piece + 2 * quad * C::kPieceStride + row;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (2 * quad + h < G) {
#pragma unroll
          for (int t = 0; t < D / 16; ++t) {
            at[h * C::kPieceStride + 16 * t] = o[t][h] * inv[h];
            at[h * C::kPieceStride + 16 * t + 8] = o[t][2 + h] * inv[h];
          }
          if (row == 0) *reinterpret_cast<float2*>(at + h * C::kPieceStride + D) = make_float2(m[h], l[h]);
        }
      }
      if (lane == 0) {
        Rec& rec = recs[warp];
        if (starts) { rec.b1 = w.b; rec.g1 = w.g; rec.u1 = w.u; }
        else { rec.b0 = w.b; rec.g0 = w.g; rec.u0 = w.u; }
      }
      flags |= starts ? kHas1 : kHas0 | (ends ? kEnds0 : 0);
    }
    walk_next(ln, w);
  }
  COOPT_TRACE_CYCLES(p.trace, kTrWarpEnd + warp, lane == 0);
  COOPT_TRACE_VALUE(p.trace, kTrBlocks, tid == 0, consumed);
  if ((cut[0] & 2u) != 0) break;         // solo: one share a CTA
  if (L == 1) {
    if (lane == 0) recs[warp].flags = flags;
    __syncthreads();
  } else {
    if (round > 0 && flags == 0 && !dead && !mbar_wait_bounded(bar_merged, (round - 1) & 1u)) dead = true;   // (its record is still in use)
    // A warp whose wait has run out leaves without another word to the others (its record may still be in use, and an arrival
    // ahead of its time would complete a phase that others have not reached): their waits for it run out in turn.
    dead = __any_sync(0xffffffffu, dead);
    if (dead) break;
    __syncwarp();                        // every lane's part of the pieces is there (a vote orders no memory)
    if (lane == 0) {
      recs[warp].flags = flags;
      mbar_arrive(bar_pieces);
    }
    dead = !mbar_wait_bounded(bar_pieces, round & 1u);
    dead = __any_sync(0xffffffffu, dead);
    if (dead) break;
  }
  COOPT_TRACE_CYCLES(p.trace, kTrStreamed, tid == 0);

  Merge<D, FMT, L> merge{p, table, ln, smem, recs, cut[1], piece0_off, piece1_off, warp, lane, y};
  merge.local(v_share);
  if (L > 1 || p.chunk_blocks == 0) {
    __syncwarp();
    if (L > 1 && lane == 0) mbar_arrive(bar_merged);
    merge.count_and_finish();
    if (L > 1) continue;
    break;
  }

  // ---- Opt-Pa: what this CTA holds of a (sequence, kv head) is merged over its chunks, then with the other CTAs' shares ----
  __syncthreads();                       // this CTA's chunks have been exported (or left in its slots)
  int task = 0;
  Walk c;
  {
    unsigned lo, hi;
    share_range(share, lo, hi);
    walk_start(ln, c, lo, hi, lane);
  }
  while (c.more) {
    const int b = c.b, g = c.g, nb = c.nb, c_first = c.u / ln.chunk;
    const bool cut_first = c.j != 0 || c.jend != c.n, first_began = c.j == 0, run_begins = first_began && c.u == 0;
    bool cut_last = false, run_ends = false;
    int c_last = c_first;
    do {
      c_last = c.u / ln.chunk;
      cut_last = c.j != 0 || c.jend != c.n;
      run_ends = c.u + c.n >= nb && c.jend == c.n;
      walk_next(ln, c);
    } while (c.more && c.b == b && c.g == g);
    // A single chunk has been stored with its export.  (16 heads over 4, head_dim 64, bf16, one sequence of 300 tokens in a chunk
    // of 2048: 14.1 us read back and merged, 11.0 so.)
    if (nb <= ln.chunk) continue;
    for (int h = 0; h < G; ++h, ++task) {
      if (task % C::kWarps != warp) continue;
      Acc a;
      acc_clear(a);
      const size_t rows = (static_cast<size_t>(b) * Hq + g * G + h) * p.max_chunks;
      auto cut = [&](int i) { return (i == c_first && cut_first) || (i == c_last && cut_last); };
      auto slot = [&](int i) { return merge.slot_of(1, share, i != c_first || first_began, h); };
      for (int c0 = c_first; c0 <= c_last; c0 += 32) {
        const int n = min(32, c_last - c0 + 1);
        float m = 0.0f, l = 0.0f;
        if (lane < n) {
          const int i = c0 + lane;
          m = cut(i) ? __ldcg(p.run_m + slot(i)) : __ldcg(p.part_m + rows + i) * kLog2e;
          l = cut(i) ? __ldcg(p.run_l + slot(i)) * kUnshift : __ldcg(p.part_l + rows + i);
        }
        acc_merge<true>(a, n, m, l, merge.on(), [&](int k) { return (cut(c0 + k) ? p.run_o + slot(c0 + k) * D : p.part_o + (rows + c0 + k) * D) + lane * 4; });
      }
      if (run_begins && run_ends) {
        merge.store_out(a, b, g, h);
      } else {
        const int u_last = (nb - 1) / ln.chunk * ln.chunk;
        const unsigned first = unit_place(ln, b, g, 0) + (whole ? 0 : kUnitCost);
        const unsigned last = unit_place(ln, b, g, u_last) + (whole ? 0 : kUnitCost + (nb - u_last) - 1);
        const int cta_f = first / T;
        merge.leave_piece(a, 0, share, run_begins, b, g, h, 0, cta_f, static_cast<int>(last / T) - cta_f + 1);
      }
    }
  }
  merge.count_and_finish();              // of chunks and of outputs together
  }
  COOPT_TRACE_CYCLES(p.trace, kTrExit, tid == 0);
  COOPT_TRACE_NS(p.trace, kTrExitNs, tid == 0);
  // a warp that gave up still has copies in flight: they get a bounded time to land
  if (dead) {
    if (lane == 0) atomicCAS(p.status, 0, COOPT_ERR_TIMEOUT);
    for (; consumed < issued; ++consumed) {
      mbar_wait_bounded(&bars[out_stage], out_phase);
      if (++out_stage == C::kStages) { out_stage = 0; out_phase ^= 1u; }
    }
  }
}

template <int D, int FMT, int L>
int launch_one(const DecodeParams& p, const LayerTable<L>& table, int grid, cudaStream_t stream) {
  using C = Cfg<D, FMT>;
  if (!configure_kernel_smem(reinterpret_cast<const void*>(&paged_decode_kernel<D, FMT, L>), C::kSmemBytes)) return COOPT_ERR_CUDA;
  return launch_dependent(paged_decode_kernel<D, FMT, L>, grid, C::kThreads, C::kSmemBytes, stream, p, table) ? COOPT_OK : COOPT_ERR_CUDA;
}

// coopt_decode_plan: a copy of the step's context lengths and of the valid part of its block table, with the block ids
// range-checked once (a bad one is replaced by 0 and reported by the launches that read the plan).  All the rest of
// the decomposition follows from the lengths, and every CTA of the attention kernel works out its own part of it.
constexpr int kPlanThreads = 256;
constexpr int kPlanPiece = 128;          // table entries a warp takes at a time
__global__ void __launch_bounds__(kPlanThreads) decode_plan_kernel(const int* block_table, int width, const int* context_lens, int batch, int num_blocks,
                                                                   int key, PlanHeader* header) {
  wait_previous_kernel();
  int* lens = reinterpret_cast<int*>(header + 1);
  int* table = reinterpret_cast<int*>(reinterpret_cast<uint8_t*>(header) + plan_table_offset(batch));
  __shared__ int bad;
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, warps = gridDim.x * (kPlanThreads / 32);
  const int per_row = (width + kPlanPiece - 1) / kPlanPiece;
  for (int i = (blockIdx.x * kPlanThreads + threadIdx.x) >> 5; i < batch * per_row; i += warps) {
    const int b = i / per_row, j0 = (i - b * per_row) * kPlanPiece + lane;
    const int L = max(0, min(context_lens[b], width * kBlockSize)), nb = (L + kBlockSize - 1) / kBlockSize;
    if (j0 == 0) lens[b] = L;
    const size_t at = static_cast<size_t>(b) * width + j0;
    int id[kPlanPiece / 32];
#pragma unroll
    for (int k = 0; k < kPlanPiece / 32; ++k) id[k] = j0 + 32 * k < nb ? block_table[at + 32 * k] : 0;
#pragma unroll
    for (int k = 0; k < kPlanPiece / 32; ++k) {
      if (id[k] < 0 || id[k] >= num_blocks) { bad = 1; id[k] = 0; }
      if (j0 + 32 * k < nb) table[at + 32 * k] = id[k];
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) header->status[blockIdx.x] = bad ? COOPT_ERR_INVALID_ARG : COOPT_OK;
  if (blockIdx.x == 0) {
    if (threadIdx.x == 0) header->key = key;
    for (int i = gridDim.x + threadIdx.x; i < kPlanCtas; i += kPlanThreads) header->status[i] = COOPT_OK;
  }
}

}  // namespace

template <int D, int FMT>
static int launch_layers(const DecodeParams& p, const coopt_layer_io* io, int grid, cudaStream_t stream) {
  auto fill = [&](LayerPtrs* l) {
    for (int y = 0; y < p.layers; ++y) {
      l[y].cache = static_cast<uint8_t*>(io[y].cache->data);
      l[y].q = static_cast<const __nv_bfloat16*>(io[y].q);
      l[y].out = static_cast<__nv_bfloat16*>(io[y].out);
      l[y].k_new = static_cast<const __nv_bfloat16*>(io[y].k_new);
      l[y].v_new = static_cast<const __nv_bfloat16*>(io[y].v_new);
      l[y].slot_mapping = reinterpret_cast<const long long*>(io[y].slot_mapping);
    }
  };
  if constexpr (FMT != COOPT_KV_BF16) {
    if (p.layers > 1) {
      LayerTable<kManyLayers> table = {};
      fill(table.l);
      return launch_one<D, FMT, kManyLayers>(p, table, grid, stream);
    }
  }
  LayerTable<1> table;
  fill(table.l);
  return launch_one<D, FMT, 1>(p, table, grid, stream);
}
static int launch_attention(const DecodeParams& p, const coopt_layer_io* io, int head_dim, int dtype, int grid, cudaStream_t stream) {
  if (head_dim == 128) {
    if (dtype == COOPT_KV_FP8_E4M3) return launch_layers<128, COOPT_KV_FP8_E4M3>(p, io, grid, stream);
    if (dtype == COOPT_KV_FP8_E5M2) return launch_layers<128, COOPT_KV_FP8_E5M2>(p, io, grid, stream);
    return launch_layers<128, COOPT_KV_BF16>(p, io, grid, stream);
  }
  if (dtype == COOPT_KV_FP8_E4M3) return launch_layers<64, COOPT_KV_FP8_E4M3>(p, io, grid, stream);
  if (dtype == COOPT_KV_FP8_E5M2) return launch_layers<64, COOPT_KV_FP8_E5M2>(p, io, grid, stream);
  return launch_layers<64, COOPT_KV_BF16>(p, io, grid, stream);
}

// Shares of a layer (the most it can have), from what the host knows: one for every CTA that fits the device, or fewer
// where even full block tables would not fill them.  The same on the sizing and the launching side.
int decode_shares(int num_sms, int batch, int num_kv_heads, int max_blocks_per_seq, int chunk_blocks) {
  const long long units = chunk_blocks > 0 ? (max_blocks_per_seq + chunk_blocks - 1) / chunk_blocks : 1;
  const long long places = static_cast<long long>(batch) * num_kv_heads * (max_blocks_per_seq + units * kUnitCost);
  const long long most = (places + kMinPlaces - 1) / kMinPlaces;
  return static_cast<int>(most < kCtasPerSm * num_sms ? most : kCtasPerSm * num_sms);
}
size_t workspace_control_bytes() { return kWsHeaderBytes + static_cast<size_t>(kCounterSlots) * 4; }
int decode_max_batch() { return kMaxBatch; }
int decode_counter_slots() { return kCounterSlots; }
int decode_max_chunk_blocks() { return kMaxChunkBlocks; }

// Workspace layout: [header 256 B: word 0 = status][counters int32 x 16384][chunk mode: exported partials][shared pieces].
void chunk_partial_offsets(int batch, int num_q_heads, int head_dim, int max_chunks, size_t* o, size_t* m, size_t* l) {
  const size_t rows = static_cast<size_t>(batch) * num_q_heads * max_chunks;
  *o = workspace_control_bytes();
  *m = *o + rows * head_dim * 4;
  *l = *m + rows * 4;
}
static size_t pieces_offset(int batch, int num_q_heads, int head_dim, int max_chunks) {
  const size_t partials = static_cast<size_t>(batch) * num_q_heads * max_chunks * (head_dim + 2) * 4;
  return (workspace_control_bytes() + partials + 255) / 256 * 256;
}
// two pieces a share: of every layer of the launch, or (chunk mode) of sequences and of chunks
static size_t pieces_rows(int shares, int group, int layers, int max_chunks) { return static_cast<size_t>(max_chunks > 0 ? 4 : 2 * layers) * shares * group; }

size_t decode_workspace_bytes(int shares, int group, int head_dim, int batch, int num_q_heads, int layers, int max_chunks) {
  return (pieces_offset(batch, num_q_heads, head_dim, max_chunks) + pieces_rows(shares, group, layers, max_chunks) * (head_dim + 2) * 4 + 255) / 256 * 256;
}
size_t decode_plan_bytes(int batch, int max_blocks_per_seq) {
  return plan_table_offset(batch) + static_cast<size_t>(batch) * max_blocks_per_seq * 4;
}

int launch_decode_plan(const int32_t* block_table, int32_t max_blocks_per_seq, const int32_t* context_lens, int32_t batch,
                       int32_t num_kv_heads, int32_t num_blocks, int32_t chunk_size, void* plan, cudaStream_t stream) {
  const long long pieces = static_cast<long long>(batch) * ((max_blocks_per_seq + kPlanPiece - 1) / kPlanPiece);
  const long long ctas = (pieces + kPlanThreads / 32 - 1) / (kPlanThreads / 32);
  const int key = plan_key(batch, num_kv_heads, chunk_size / kBlockSize, max_blocks_per_seq, num_blocks);
  return launch_dependent(decode_plan_kernel, static_cast<int>(ctas < kPlanCtas ? ctas : kPlanCtas), kPlanThreads, 0, stream, block_table,
                          max_blocks_per_seq, context_lens, batch, num_blocks, key, static_cast<PlanHeader*>(plan))
             ? COOPT_OK
             : COOPT_ERR_CUDA;
}

int launch_decode(const DecodeCall& a, cudaStream_t stream) {
  const coopt_cache* c = a.layers[0].cache;            // all of one shape
  DecodeParams p = {};
  p.layers = a.num_layers;
  p.shares = a.shares;
  p.block_table = a.block_table;
  p.context_lens = a.context_lens;
  p.cu_q_lens = a.cu_q_lens;
  p.max_blocks_per_seq = a.max_blocks_per_seq;
  p.batch = a.batch;
  p.num_q_heads = a.num_q_heads;
  p.num_kv_heads = c->num_kv_heads;
  p.group = a.num_q_heads / c->num_kv_heads;
  p.num_blocks = c->num_blocks;
  p.solo_blocks = std::max(kSoloUnits, std::min(kSoloMost, a.batch * c->num_kv_heads / kSoloShare));
  p.sm_scale_log2 = a.sm_scale * kLog2e;
  p.chunk_blocks = a.chunk_size / kBlockSize;
  p.max_chunks = a.chunk_size > 0 ? static_cast<int>((static_cast<long long>(a.max_blocks_per_seq) * kBlockSize + a.chunk_size - 1) / a.chunk_size) : 0;
  if (a.plan != nullptr) {
    const uint8_t* plan = static_cast<const uint8_t*>(a.plan);
    p.plan = reinterpret_cast<const PlanHeader*>(plan);
    p.context_lens = reinterpret_cast<const int*>(plan + kPlanHeaderBytes);
    p.block_table = reinterpret_cast<const int*>(plan + plan_table_offset(a.batch));
    p.plan_key = plan_key(a.batch, c->num_kv_heads, p.chunk_blocks, a.max_blocks_per_seq, c->num_blocks);
  }
  p.kv_token_stride = a.kv_token_stride;
  p.order = a.order;
  uint8_t* ws = static_cast<uint8_t*>(a.workspace);
  p.status = reinterpret_cast<int*>(ws);
  p.counters = reinterpret_cast<int*>(ws + kWsHeaderBytes);
  if (a.chunk_size > 0) {
    size_t o, m, l;
    chunk_partial_offsets(a.batch, a.num_q_heads, c->head_dim, p.max_chunks, &o, &m, &l);
    p.part_o = reinterpret_cast<float*>(ws + o);
    p.part_m = reinterpret_cast<float*>(ws + m);
    p.part_l = reinterpret_cast<float*>(ws + l);
  }
  const size_t rows = pieces_rows(a.shares, p.group, a.num_layers, p.max_chunks);
  p.run_o = reinterpret_cast<float*>(ws + pieces_offset(a.batch, a.num_q_heads, c->head_dim, p.max_chunks));
  p.run_m = p.run_o + rows * c->head_dim;
  p.run_l = p.run_m + rows;
#ifdef COOPT_TRACE
  p.trace = trace_buffer();
#endif
  return launch_attention(p, a.layers, c->head_dim, c->dtype, std::min(kCtasPerSm * a.num_sms, a.shares * a.num_layers), stream);
}

}  // namespace coopt
