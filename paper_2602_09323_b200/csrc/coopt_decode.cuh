// Paged GQA decode: what the kernel and the host side share: the work decomposition, the layout of a plan buffer and
// the kernel's parameters.
//
// Work decomposition (Eq. 9: only the valid blocks of every sequence are listed).  A unit is what one softmax runs
// over before anything is merged: a (sequence, kv head), or in chunk mode (Opt-Pa) one chunk of one.  All units of a layer
// lie one behind the other on a line, in the order sequence, kv head, chunk; a unit of n blocks takes n + kUnitCost places
// of it, the extra ones in front, because a unit costs its warp a start and an end (query rows, reduction, store)
// besides its blocks.  Share i of the line has the places [i T, (i + 1) T); a CTA works through one share, or through one
// of every layer; warp w takes an equal part of the share's places, and a block belongs to the warp that holds its place.
// So every warp has at most two units of a share that it holds only a piece of: the one it starts in the middle of, and
// the one it does not reach the end of.
#pragma once

#include "coopt_common.cuh"

namespace coopt {

constexpr int kMaxBatch = 512;
constexpr int kMaxGroup = 8;
constexpr int kMaxChunkBlocks = 2048;
constexpr int kCounterSlots = 16384;  // >= kManyLayers * shares * kMaxGroup
constexpr int kWsHeaderBytes = 256;
// Measured, us a pass: cost 3 / 5 / 8 places 391 / 394 / 390 (64 mixed lengths, 4 layers), 125 / 123 / 121 (24 sequences, G = 8,
// 4 layers), 235.5 / 231.5 / 239.8 (32 x 2048 tokens, 8 layers); smallest share 8 / 16 / 64 places 12.2 / 12.3 / 16.6 (one
// sequence of 777 tokens), 11.9 / 11.6 / 15.2 (one of 2000), 13.7 / 13.6 / 15.3 (four of 1600..3000), 20.6 / 20.6 / 18.0 (7 of
// 272..544 tokens, 8 layers): where a call cannot fill the device, spreading it wins, except in launches over several layers.
constexpr int kUnitCost = 5;          // places of the line that a unit takes besides its blocks
constexpr int kCtasPerSm = 1;
constexpr int kMinPlaces = 16;        // smallest share
// Units of at most so many blocks at head_dim 64, half as many at 128, are not cut between shares.  (Device full, not cut / cut:
// 64 sequences of up to 16 and 24 blocks, 40 heads over 8, head_dim 128 15.4 / 16.7 and 16.6 / 18.2 us; 130 of up to 32, 16 over
// 4, head_dim 64 15.5 / 17.2.)
constexpr int kWholeUnits = 32;
// .. where the call does not fill the device.  One layer alone would have the line at 40 blocks (one sequence, 40 heads over 8,
// head_dim 128, 32 / 48 / 96 blocks: 10.2 / 11.8 / 16.0 us not cut, 10.5 / 10.5 / 10.9 cut; head_dim 64, 32 / 48 / 96 / 192: 9.2 /
// 10.3 / 13.4 / 18.4 and 10.3 / 10.3 / 10.9 / 11.9), but a layer is cut the same way alone and in a launch over several, where
// units that are not cut win throughout (eight layers of four sequences of 64 blocks 25.5 / 77.9; of one of 96 17.4 / 32.2).
constexpr int kWholeUnitsIdle = 192;
// .. and of a bf16 cache, which has no launch over several layers: blocks at either head dim.  (One sequence, 8 heads, head_dim
// 128, 32 / 48 / 64 blocks: 9.0 / 10.5 / 11.8 us not cut, 9.4 / 9.6 / 10.2 cut; head_dim 64: 8.6 / 9.7 / 10.8 and 9.0 / 9.3 / 10.0.)
constexpr int kWholeUnitsIdleBf16 = 40;
// Units of at most so many blocks are not cut between warps either.  Eight layers of 40 sequences, 4 kv heads, us against units
// spread over a CTA's warps: 1 block 10.6 / 27.6, 4 blocks 13.6 / 44, 8 blocks 17.5 / 65; one layer: 8.8 / 8.8, 11.7 / 10.5,
// 14.0 / 10.5.
constexpr int kSoloUnits = 4;
// .. or of more, the more units there are to keep the warps busy: one block for every kSoloShare units, at most kSoloMost.
// (Four kv heads, eight layers / one, cut between warps and not: 160 sequences of 10 blocks 112 / 16.5 and 53 / 16.9 us, 400 of
// 10 blocks 181 / 26.5 and 126 / 22.2, 400 of 1..16 blocks 175 / 25.8 and 112 / 30.0, 80 of 12 blocks 96 / 14.2 and 41 / 19.8.)
constexpr int kSoloShare = 48, kSoloMost = 12;
constexpr int kNoChunks = 1 << 30;    // "blocks per chunk" of a call without chunks

// A plan: header, the clamped context lengths int32[batch] (padded to 16 bytes), the block table
// int32[batch][max_blocks_per_seq] with its valid entries range-checked.
constexpr int kPlanCtas = 48;
struct PlanHeader {
  int key;                   // plan_key() of the problem the plan was made for
  int pad[15];
  int status[kPlanCtas];     // by CTA of the planning kernel: a coopt_status that the launches which read the plan report
};
constexpr int kPlanHeaderBytes = 256;
static_assert(sizeof(PlanHeader) == kPlanHeaderBytes, "plan layout");
__host__ __device__ inline size_t plan_table_offset(int batch) { return kPlanHeaderBytes + (static_cast<size_t>(batch) * 4 + 15) / 16 * 16; }

// What a launch and the plan it is handed must agree on.
__host__ __device__ inline int plan_key(int batch, int num_kv_heads, int chunk_blocks, int max_blocks_per_seq, int num_blocks) {
  unsigned int h = 0x9e3779b9u;
  const int v[5] = {batch, num_kv_heads, chunk_blocks, max_blocks_per_seq, num_blocks};
  for (int i = 0; i < 5; ++i) h = (h ^ static_cast<unsigned int>(v[i])) * 0x01000193u + 0x7f4a7c15u;
  return static_cast<int>(h | 1u);
}

// What a layer brings of its own.
struct LayerPtrs {
  uint8_t* cache;
  const __nv_bfloat16* q;
  __nv_bfloat16* out;
  // fused append (null when the layer has no new tokens): Algorithm 1 phase 1 for one token per sequence
  const __nv_bfloat16* k_new;
  const __nv_bfloat16* v_new;
  const long long* slot_mapping;
};
// A launch serves one layer, or up to kManyLayers of any size whose buffers do not touch each other (every one has room of its
// own for its pieces in the workspace; what a launch costs once is small against eight layers).
constexpr int kManyLayers = 8;
template <int L>
struct LayerTable {
  LayerPtrs l[L];
};

struct DecodeParams {
  const int* block_table;
  const int* context_lens;
  const PlanHeader* plan;  // null: block_table and context_lens are the caller's own and are checked here
  const int* cu_q_lens;    // chunk mode of coopt_paged_chunked: prefix sums of the query tokens (must be 0..batch); else null
  int plan_key;
  long long kv_token_stride;
  int layers;
  int shares;              // decode_shares(): the most shares a layer can have
  int max_blocks_per_seq;
  int batch, num_q_heads, num_kv_heads, group;
  int num_blocks;
  int solo_blocks;         // units of at most so many blocks are held whole by a warp
  int order;               // DecodeOrder
  float sm_scale_log2;     // sm_scale * log2(e)
  int chunk_blocks;        // 0 = decode mode
  int max_chunks;
  int* status;
  int* counters;           // [regions][shares][kMaxGroup]: pieces delivered, by first share and head
  float* part_o;           // chunk mode: exported partials [B][Hq][max_chunks][D]
  float* part_m;           // [B][Hq][max_chunks]
  float* part_l;
  float* run_o;            // pieces of units that are cut between shares: [regions][2 shares][G][D]; a region per layer, or (chunk
                           // mode) region 0 for (sequence, kv head), region 1 for chunks
  float* run_m;            // [regions][2 shares][G], base-2 logarithm units
  float* run_l;
  unsigned long long* trace;   // time stamps (trace build only; null otherwise)
};

// ---- host side -------------------------------------------------------------------------------------------------
// How much of a launch may run while the kernel in front of it in the stream still does.
enum DecodeOrder {
  kDependent,             // nothing but set-up
  kAfterWrite,            // lengths and block table (or plan) were complete before that kernel began: they are read early
  kOverlapPrevious        // .. and so was the cache: its first blocks are requested early
};
struct DecodeCall {
  const coopt_layer_io* layers;
  int32_t num_layers;               // <= kManyLayers
  const int32_t* block_table;       // these two, or a plan
  const int32_t* context_lens;
  const void* plan;
  const int32_t* cu_q_lens;
  int64_t kv_token_stride;
  int32_t max_blocks_per_seq, batch, num_q_heads, chunk_size;
  float sm_scale;
  void* workspace;
  int shares;                       // decode_shares()
  int num_sms;
  DecodeOrder order;
};
int launch_decode(const DecodeCall& a, cudaStream_t stream);
int launch_decode_plan(const int32_t* block_table, int32_t max_blocks_per_seq, const int32_t* context_lens, int32_t batch,
                       int32_t num_kv_heads, int32_t num_blocks, int32_t chunk_size, void* plan, cudaStream_t stream);
int decode_shares(int num_sms, int batch, int num_kv_heads, int max_blocks_per_seq, int chunk_blocks);
size_t decode_workspace_bytes(int shares, int group, int head_dim, int batch, int num_q_heads, int layers, int max_chunks);
size_t decode_plan_bytes(int batch, int max_blocks_per_seq);
size_t workspace_control_bytes();
size_t workspace_need(int batch, int num_q_heads, int num_kv_heads, int head_dim, int max_blocks_per_seq, int chunk_size, int layers);
int decode_max_batch();
int decode_counter_slots();
int decode_max_chunk_blocks();
void chunk_partial_offsets(int batch, int num_q_heads, int head_dim, int max_chunks, size_t* o, size_t* m, size_t* l);

}  // namespace coopt
