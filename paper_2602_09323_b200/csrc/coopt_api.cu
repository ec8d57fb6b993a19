// Host side of the C ABI: argument checks, workspace arithmetic, dispatch to the launchers.
#include <algorithm>
#include <mutex>
#include <utility>
#include <vector>

#include "coopt_decode.cuh"

namespace coopt {

int launch_kv_write(const coopt_cache* c, const void* k, const void* v, int64_t stride, const int64_t* slots,
                    int num_tokens, cudaStream_t stream);
int launch_paged_prefill(const coopt_cache* c, const void* q, void* out, const int32_t* cu_q_lens,
                         const int32_t* block_table, int32_t max_blocks_per_seq, const int32_t* context_lens,
                         int32_t batch, int32_t num_q_heads, int32_t total_q, int32_t causal, float sm_scale,
                         void* workspace, int num_sms, cudaStream_t stream);
const DeviceInfo* device_info() {
  static DeviceInfo info[64];
  static bool known[64] = {};
  static std::mutex mu;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  std::lock_guard<std::mutex> lock(mu);
  if (!known[dev]) {
    int sms = 0, smem = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return nullptr;
    if (cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) return nullptr;
    info[dev].num_sms = sms;
    info[dev].max_smem_optin = smem;
    known[dev] = true;
  }
  return &info[dev];
}

bool configure_kernel_smem(const void* kernel, int bytes) {
  static std::mutex mu;
  static std::vector<std::pair<const void*, int>> done;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  std::lock_guard<std::mutex> lock(mu);
  for (const auto& d : done)
    if (d.first == kernel && d.second == dev) return true;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return false;
  done.emplace_back(kernel, dev);
  return true;
}

namespace {

bool cache_shape_ok(int head_dim, int block_size, int dtype) {
  return (head_dim == 64 || head_dim == 128) && block_size == kBlockSize &&
         (is_fp8(dtype) || dtype == COOPT_KV_BF16);
}

int check_cache(const coopt_cache* c) {
  if (c == nullptr || c->data == nullptr || c->num_blocks <= 0 || c->num_kv_heads <= 0) return COOPT_ERR_INVALID_ARG;
  if (!cache_shape_ok(c->head_dim, c->block_size, c->dtype)) return COOPT_ERR_UNSUPPORTED;
  if (reinterpret_cast<uintptr_t>(c->data) % 32 != 0) return COOPT_ERR_INVALID_ARG;
  return COOPT_OK;
}

int max_chunks_of(int max_blocks_per_seq, int chunk_size) {
  return static_cast<int>((static_cast<long long>(max_blocks_per_seq) * kBlockSize + chunk_size - 1) / chunk_size);
}

int num_sms() {
  const DeviceInfo* di = device_info();
  return std::min(di ? di->num_sms : 148, kCounterSlots / (kManyLayers * kMaxGroup) / kCtasPerSm);
}
int shares_of(int batch, int num_kv_heads, int max_blocks_per_seq, int chunk_size) {
  return decode_shares(num_sms(), batch, num_kv_heads, max_blocks_per_seq, chunk_size / kBlockSize);
}

// The sizes that coopt_plan_bytes and coopt_workspace_bytes report are part of the interface: pools are laid out by them,
// and coopt_paged_decode_static refuses by them.  They are those of a plan that lists every CTA's blocks and of a
// workspace with room for one -- more than the kernels use now, except for the pieces of small problems.
long long listed_plan_ctas(int batch, int num_kv_heads, int max_blocks_per_seq) {
  const DeviceInfo* di = device_info();
  const long long sms = di ? di->num_sms : 148, need = (static_cast<long long>(batch) * num_kv_heads * max_blocks_per_seq + 2031) / 2032;
  return need > sms ? need : sms;
}
size_t listed_plan_bytes(int batch, int num_kv_heads, int max_blocks_per_seq, int chunk_blocks) {
  const long long P = listed_plan_ctas(batch, num_kv_heads, max_blocks_per_seq);
  const long long units = static_cast<long long>(batch) * num_kv_heads, all = units * max_blocks_per_seq;
  long long blocks = (all + P - 1) / P + 1;
  if (chunk_blocks > 0) {
    const long long chunks = units * ((max_blocks_per_seq + chunk_blocks - 1) / chunk_blocks);
    blocks = ((chunks + P - 1) / P + 1) * chunk_blocks;
  } else if (blocks < 32) {
    blocks = 32;
  }
  if (blocks > all) blocks = all;
  long long segments = (blocks < units ? blocks : units) + 3;
  if (chunk_blocks > 0) segments += blocks / chunk_blocks + 1;
  if (segments > blocks + 2) segments = blocks + 2;
  const long long rounds = (segments + 31) / 32 + (blocks + 1023) / 1024 + 1;
  const long long region = (rounds * 80 + segments * 64 + blocks * 4 + 64 + 127) / 128 * 128;
  return 256 + static_cast<size_t>(P) * region + 4096;
}
size_t larger(size_t a, size_t b) { return a > b ? a : b; }

}  // namespace

// What a call over that many layers has to be given.
size_t workspace_need(int batch, int num_q_heads, int num_kv_heads, int head_dim, int max_blocks_per_seq, int chunk_size, int layers) {
  const int group = (num_q_heads + num_kv_heads - 1) / num_kv_heads;
  const int mc = chunk_size > 0 ? max_chunks_of(max_blocks_per_seq, chunk_size) : 0;
  const size_t used = decode_workspace_bytes(shares_of(batch, num_kv_heads, max_blocks_per_seq, chunk_size), group, head_dim, batch, num_q_heads, layers, mc);
  const size_t pieces = static_cast<size_t>(2) * listed_plan_ctas(batch, num_kv_heads, max_blocks_per_seq) * group * (head_dim + 2) * 4;
  const size_t partials = static_cast<size_t>(batch) * num_q_heads * mc * (head_dim + 2) * 4;
  const size_t listed = (workspace_control_bytes() + pieces + (mc > 0 ? partials + 256 : 0) + 511) / 256 * 256 +
                        listed_plan_bytes(batch, num_kv_heads, max_blocks_per_seq, chunk_size / kBlockSize);
  return larger(used, listed);
}

int check_attention_shapes(const coopt_cache* c, const void* q, void* out, int32_t max_blocks_per_seq, int32_t batch,
                           int32_t num_q_heads);

// Every host-side check of a decode-style call (shared with the entry points of other files).
int check_attention_args(const coopt_cache* c, const void* q, void* out, const int32_t* block_table,
                         int32_t max_blocks_per_seq, const int32_t* context_lens, int32_t batch, int32_t num_q_heads) {
  const int rc = check_attention_shapes(c, q, out, max_blocks_per_seq, batch, num_q_heads);
  if (rc != COOPT_OK) return rc;
  return block_table && context_lens ? COOPT_OK : COOPT_ERR_INVALID_ARG;
}

int check_attention_shapes(const coopt_cache* c, const void* q, void* out, int32_t max_blocks_per_seq, int32_t batch,
                           int32_t num_q_heads) {
  const int rc = check_cache(c);
  if (rc != COOPT_OK) return rc;
  if (!q || !out || batch < 0 || max_blocks_per_seq <= 0 || num_q_heads <= 0) return COOPT_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(q) | reinterpret_cast<uintptr_t>(out)) % 16 != 0) return COOPT_ERR_INVALID_ARG;   // rows move in 16-byte pieces
  if (num_q_heads % c->num_kv_heads != 0) return COOPT_ERR_UNSUPPORTED;
  const int group = num_q_heads / c->num_kv_heads;
  if (group < 1 || group > 8) return COOPT_ERR_UNSUPPORTED;
  if (batch > decode_max_batch() || static_cast<long long>(batch) * c->num_kv_heads > decode_counter_slots())
    return COOPT_ERR_UNSUPPORTED;
  // the planner indexes (sequence, kv head, block) triples with 31 bits
  if (static_cast<long long>(batch) * c->num_kv_heads * max_blocks_per_seq >= (1ll << 31)) return COOPT_ERR_UNSUPPORTED;
  return COOPT_OK;
}

// What every decode-style launch has in common.
static DecodeCall attention_call(const coopt_layer_io* layers, int32_t num_layers, int32_t max_blocks_per_seq, int32_t batch, int32_t num_q_heads,
                                 int32_t chunk_size, float sm_scale, void* workspace) {
  DecodeCall a = {};
  a.layers = layers;
  a.num_layers = num_layers;
  a.max_blocks_per_seq = max_blocks_per_seq;
  a.batch = batch;
  a.num_q_heads = num_q_heads;
  a.chunk_size = chunk_size;
  a.sm_scale = sm_scale;
  a.workspace = workspace;
  a.num_sms = num_sms();
  a.shares = shares_of(batch, layers[0].cache->num_kv_heads, max_blocks_per_seq, chunk_size);
  a.order = kDependent;
  return a;
}

// Whether layers may run side by side: nothing that one of them writes (its output; its cache if it appends) is read or
// written by another, nor read by all (block table, context lengths).
static bool layers_are_apart(const coopt_layer_io* layers, int num_layers, int64_t kv_token_stride, const int32_t* block_table, int max_blocks_per_seq,
                             const int32_t* context_lens, int batch, int num_q_heads) {
  struct Range { uintptr_t lo, hi; int layer; bool write; };
  Range r[6 * kManyLayers + 2];
  int n = 0;
  auto add = [&](const void* p, size_t bytes, int layer, bool write) {
    if (p != nullptr && bytes > 0) r[n++] = Range{reinterpret_cast<uintptr_t>(p), reinterpret_cast<uintptr_t>(p) + bytes, layer, write};
  };
  const coopt_cache& c = *layers[0].cache;
  const size_t rows = static_cast<size_t>(batch) * num_q_heads * c.head_dim * 2;
  const size_t cache = static_cast<size_t>(c.num_blocks) * c.num_kv_heads * granule_bytes(c.head_dim, true);
  const size_t tokens = (static_cast<size_t>(batch - 1) * kv_token_stride + static_cast<size_t>(c.num_kv_heads) * c.head_dim) * 2;
  for (int y = 0; y < num_layers; ++y) {
    const coopt_layer_io& io = layers[y];
    add(io.q, rows, y, false);
    add(io.out, rows, y, true);
    add(io.cache->data, cache, y, io.k_new != nullptr);
    add(io.k_new, tokens, y, false);
    add(io.v_new, tokens, y, false);
    add(io.slot_mapping, static_cast<size_t>(batch) * 8, y, false);
  }
  add(block_table, static_cast<size_t>(batch) * max_blocks_per_seq * 4, -1, false);
  add(context_lens, static_cast<size_t>(batch) * 4, -1, false);
  std::sort(r, r + n, [](const Range& a, const Range& b) { return a.lo < b.lo; });
  // in order of their begins: how far the ranges before reach, by the layer that reaches farthest and by the others
  struct Reach {
    uintptr_t hi = 0, other = 0;
    int layer = -2;
    void add(const Range& x) {
      if (x.layer == layer) hi = x.hi > hi ? x.hi : hi;
      else if (x.hi > hi) { other = hi; hi = x.hi; layer = x.layer; }
      else if (x.hi > other) other = x.hi;
    }
    bool meets(const Range& x) const { return x.lo < (x.layer == layer ? other : hi); }
  } all, written;
  for (int i = 0; i < n; ++i) {
    if ((r[i].write ? all : written).meets(r[i])) return false;
    all.add(r[i]);
    if (r[i].write) written.add(r[i]);
  }
  return true;
}

// Layers that the next launch of a coopt_decode_layers call takes, of `left` (of one shape, the first of the call if `first`),
// and whether it may begin ahead of the kernel before it (the planning kernel, if it is the call's first).
struct LayersLaunch {
  int layers;
  bool early;
};
static LayersLaunch next_layers(const coopt_layer_io* layers, int left, bool first, int64_t kv_token_stride, const int32_t* block_table,
                                int max_blocks_per_seq, const int32_t* context_lens, int batch, int num_q_heads, size_t workspace_bytes, bool overlap) {
  const coopt_cache& c = *layers[0].cache;
  // Layers whose buffers are apart go into one launch, up to eight: what a launch costs once is then shared, and the pieces of a
  // layer are merged while the blocks of the next are under way.  (Apart / together, us: eight layers of 8 sequences of 1..28
  // tokens 71 / 10.1; three of 54 of 4072..8144, G = 2, 185 / 174; four of 24 of 300..4000, G = 8, 101.5 / 89.4; four of 32 x
  // 8192, G = 6, 7 and 8, 374 / 358, 376 / 359 and 377 / 360; head_dim 64, 64 of 100..5000, G = 4, four layers of eight kv heads
  // 153.5 / 141.9, eight layers of four 203 / 181.)
  int n = std::min(left, kManyLayers);
  while (n > 1 && workspace_bytes < workspace_need(batch, num_q_heads, c.num_kv_heads, c.head_dim, max_blocks_per_seq, 0, n)) --n;
  auto apart = [&](int n) { return layers_are_apart(layers, n, kv_token_stride, block_table, max_blocks_per_seq, context_lens, batch, num_q_heads); };
  if (n > 1 && !apart(n)) n = 1;
  return {n, first ? n > 1 || apart(1) : overlap};
}

}  // namespace coopt

using namespace coopt;

extern "C" {

size_t coopt_granule_bytes(int32_t head_dim, int32_t dtype) {
  if (!cache_shape_ok(head_dim, kBlockSize, dtype)) return 0;
  return granule_bytes(head_dim, is_fp8(dtype));
}

size_t coopt_cache_bytes(int32_t num_blocks, int32_t num_kv_heads, int32_t head_dim, int32_t dtype) {
  if (num_blocks <= 0 || num_kv_heads <= 0) return 0;
  return static_cast<size_t>(num_blocks) * num_kv_heads * coopt_granule_bytes(head_dim, dtype);
}

int64_t coopt_cache_offset(const coopt_cache* c, int32_t block, int32_t kv_head, int32_t which, int32_t token,
                           int32_t dim) {
  if (!c || !cache_shape_ok(c->head_dim, c->block_size, c->dtype)) return -1;
  if (block < 0 || block >= c->num_blocks || kv_head < 0 || kv_head >= c->num_kv_heads || which < 0 || which > 1 ||
      token < 0 || token >= kBlockSize || dim < 0 || dim >= c->head_dim)
    return -1;
  const bool fp8 = is_fp8(c->dtype);
  const int64_t gran = (static_cast<int64_t>(block) * c->num_kv_heads + kv_head) * granule_bytes(c->head_dim, fp8);
  const int inner = which == 0 ? k_elem_offset(c->head_dim, fp8, token, dim) : v_elem_offset(c->head_dim, fp8, token, dim);
  return gran + part_offset(c->head_dim, fp8, which) + inner;
}

int64_t coopt_scale_offset(const coopt_cache* c, int32_t block, int32_t kv_head, int32_t which) {
  if (!c || !cache_shape_ok(c->head_dim, c->block_size, c->dtype) || !is_fp8(c->dtype)) return -1;
  if (block < 0 || block >= c->num_blocks || kv_head < 0 || kv_head >= c->num_kv_heads || which < 0 || which > 1) return -1;
  return (static_cast<int64_t>(block) * c->num_kv_heads + kv_head) * granule_bytes(c->head_dim, true) + header_offset(c->head_dim) + 4 * which;
}

int coopt_kv_write(const coopt_cache* cache, const void* k, const void* v, int64_t kv_token_stride,
                   const int64_t* slot_mapping, int32_t num_tokens, void* stream) {
  const int rc = check_cache(cache);
  if (rc != COOPT_OK) return rc;
  if (num_tokens < 0) return COOPT_ERR_INVALID_ARG;
  if (num_tokens == 0) return COOPT_OK;
  if (!k || !v || !slot_mapping) return COOPT_ERR_INVALID_ARG;
  if (kv_token_stride < static_cast<int64_t>(cache->num_kv_heads) * cache->head_dim) return COOPT_ERR_INVALID_ARG;
  return launch_kv_write(cache, k, v, kv_token_stride, slot_mapping, num_tokens, static_cast<cudaStream_t>(stream));
}

size_t coopt_workspace_bytes(int32_t batch, int32_t num_q_heads, int32_t num_kv_heads, int32_t head_dim,
                             int32_t max_blocks_per_seq, int32_t chunk_size, int32_t total_q) {
  (void)total_q;
  if (batch < 0 || num_q_heads <= 0 || num_kv_heads <= 0 || max_blocks_per_seq <= 0 || chunk_size < 0) return 0;
  return larger(workspace_need(batch, num_q_heads, num_kv_heads, head_dim, max_blocks_per_seq, chunk_size, 1),
                chunk_size > 0 ? 0 : workspace_need(batch, num_q_heads, num_kv_heads, head_dim, max_blocks_per_seq, 0, kManyLayers));
}

int coopt_workspace_init(void* workspace, size_t workspace_bytes, void* stream) {
  if (!workspace) return COOPT_ERR_INVALID_ARG;
  if (workspace_bytes < workspace_control_bytes()) return COOPT_ERR_WORKSPACE;
  return cudaMemsetAsync(workspace, 0, workspace_control_bytes(), static_cast<cudaStream_t>(stream)) == cudaSuccess
             ? COOPT_OK
             : COOPT_ERR_CUDA;
}

int coopt_chunk_partials(int32_t batch, int32_t num_q_heads, int32_t head_dim, int32_t max_blocks_per_seq,
                         int32_t chunk_size, size_t* o_offset, size_t* m_offset, size_t* l_offset, int32_t* max_chunks) {
  if (batch < 0 || num_q_heads <= 0 || head_dim <= 0 || max_blocks_per_seq <= 0 || chunk_size <= 0 ||
      chunk_size % kBlockSize != 0 || !o_offset || !m_offset || !l_offset || !max_chunks)
    return COOPT_ERR_INVALID_ARG;
  *max_chunks = max_chunks_of(max_blocks_per_seq, chunk_size);
  chunk_partial_offsets(batch, num_q_heads, head_dim, *max_chunks, o_offset, m_offset, l_offset);
  return COOPT_OK;
}

int coopt_paged_decode(const coopt_cache* cache, const void* q, void* out, const int32_t* block_table,
                       int32_t max_blocks_per_seq, const int32_t* context_lens, int32_t batch, int32_t num_q_heads,
                       float sm_scale, void* workspace, size_t workspace_bytes, void* stream) {
  const int rc = check_attention_args(cache, q, out, block_table, max_blocks_per_seq, context_lens, batch, num_q_heads);
  if (rc != COOPT_OK) return rc;
  if (batch == 0) return COOPT_OK;
  if (!workspace || workspace_bytes < workspace_need(batch, num_q_heads, cache->num_kv_heads, cache->head_dim, max_blocks_per_seq, 0, 1))
    return COOPT_ERR_WORKSPACE;
  const coopt_layer_io io = {cache, nullptr, nullptr, nullptr, q, out};
  DecodeCall a = attention_call(&io, 1, max_blocks_per_seq, batch, num_q_heads, 0, sm_scale, workspace);
  a.block_table = block_table;
  a.context_lens = context_lens;
  return launch_decode(a, static_cast<cudaStream_t>(stream));
}

int coopt_decode_step(const coopt_cache* cache, const void* k_new, const void* v_new, int64_t kv_token_stride,
                      const int64_t* slot_mapping, const void* q, void* out, const int32_t* block_table,
                      int32_t max_blocks_per_seq, const int32_t* context_lens, int32_t batch, int32_t num_q_heads,
                      float sm_scale, void* workspace, size_t workspace_bytes, void* stream) {
  // every check of both halves before anything is launched
  int rc = check_attention_args(cache, q, out, block_table, max_blocks_per_seq, context_lens, batch, num_q_heads);
  if (rc != COOPT_OK) return rc;
  if (!k_new || !v_new || !slot_mapping || kv_token_stride < static_cast<int64_t>(cache->num_kv_heads) * cache->head_dim)
    return COOPT_ERR_INVALID_ARG;
  if (batch == 0) return COOPT_OK;
  if (!workspace || workspace_bytes < workspace_need(batch, num_q_heads, cache->num_kv_heads, cache->head_dim, max_blocks_per_seq, 0, 1))
    return COOPT_ERR_WORKSPACE;
  rc = launch_kv_write(cache, k_new, v_new, kv_token_stride, slot_mapping, batch, static_cast<cudaStream_t>(stream));
  if (rc != COOPT_OK) return rc;
  const coopt_layer_io io = {cache, nullptr, nullptr, nullptr, q, out};
  DecodeCall a = attention_call(&io, 1, max_blocks_per_seq, batch, num_q_heads, 0, sm_scale, workspace);
  a.block_table = block_table;
  a.context_lens = context_lens;
  a.order = kAfterWrite;
  return launch_decode(a, static_cast<cudaStream_t>(stream));
}

size_t coopt_plan_bytes(int32_t batch, int32_t num_kv_heads, int32_t max_blocks_per_seq, int32_t chunk_size) {
  if (batch <= 0 || num_kv_heads <= 0 || max_blocks_per_seq <= 0 || chunk_size < 0 || chunk_size % kBlockSize != 0) return 0;
  return larger(decode_plan_bytes(batch, max_blocks_per_seq), listed_plan_bytes(batch, num_kv_heads, max_blocks_per_seq, chunk_size / kBlockSize));
}

static int check_plan_args(int32_t batch, int32_t num_kv_heads, int32_t max_blocks_per_seq, int32_t chunk_size, const void* plan,
                           size_t plan_bytes_given) {
  if (batch < 0 || num_kv_heads <= 0 || max_blocks_per_seq <= 0) return COOPT_ERR_INVALID_ARG;
  if (chunk_size < 0 || chunk_size % kBlockSize != 0 || chunk_size / kBlockSize > decode_max_chunk_blocks()) return COOPT_ERR_INVALID_ARG;
  if (batch > decode_max_batch() || static_cast<long long>(batch) * num_kv_heads > decode_counter_slots()) return COOPT_ERR_UNSUPPORTED;
  if (static_cast<long long>(batch) * num_kv_heads * max_blocks_per_seq >= (1ll << 31)) return COOPT_ERR_UNSUPPORTED;
  if (batch == 0) return COOPT_OK;
  if (!plan || reinterpret_cast<uintptr_t>(plan) % 16 != 0) return COOPT_ERR_INVALID_ARG;
  if (plan_bytes_given < coopt_plan_bytes(batch, num_kv_heads, max_blocks_per_seq, chunk_size)) return COOPT_ERR_WORKSPACE;
  return COOPT_OK;
}

int coopt_decode_plan(const int32_t* block_table, int32_t max_blocks_per_seq, const int32_t* context_lens, int32_t batch,
                      int32_t num_kv_heads, int32_t num_blocks, int32_t chunk_size, void* plan, size_t plan_bytes_given,
                      void* stream) {
  const int rc = check_plan_args(batch, num_kv_heads, max_blocks_per_seq, chunk_size, plan, plan_bytes_given);
  if (rc != COOPT_OK) return rc;
  if (!block_table || !context_lens || num_blocks <= 0) return COOPT_ERR_INVALID_ARG;
  if (batch == 0) return COOPT_OK;
  return launch_decode_plan(block_table, max_blocks_per_seq, context_lens, batch, num_kv_heads, num_blocks, chunk_size, plan,
                            static_cast<cudaStream_t>(stream));
}

int coopt_decode_step_planned(const coopt_cache* cache, const void* plan, size_t plan_bytes_given, const void* k_new,
                              const void* v_new, int64_t kv_token_stride, const int64_t* slot_mapping, const void* q, void* out,
                              int32_t max_blocks_per_seq, int32_t batch, int32_t num_q_heads, int32_t chunk_size, float sm_scale,
                              void* workspace, size_t workspace_bytes, uint32_t flags, void* stream) {
  int rc = check_attention_shapes(cache, q, out, max_blocks_per_seq, batch, num_q_heads);
  if (rc != COOPT_OK) return rc;
  if (!is_fp8(cache->dtype)) return COOPT_ERR_UNSUPPORTED;                     // the bf16 ablation kernel plans for itself
  rc = check_plan_args(batch, cache->num_kv_heads, max_blocks_per_seq, chunk_size, plan, plan_bytes_given);
  if (rc != COOPT_OK) return rc;
  const bool append = k_new || v_new || slot_mapping;
  if (append && (!k_new || !v_new || !slot_mapping || kv_token_stride < static_cast<int64_t>(cache->num_kv_heads) * cache->head_dim))
    return COOPT_ERR_INVALID_ARG;
  if ((flags & ~static_cast<uint32_t>(COOPT_FLAG_OVERLAP_PREVIOUS)) != 0) return COOPT_ERR_INVALID_ARG;
  if (batch == 0) return COOPT_OK;
  if (!workspace || workspace_bytes < workspace_need(batch, num_q_heads, cache->num_kv_heads, cache->head_dim, max_blocks_per_seq, chunk_size, 1))
    return COOPT_ERR_WORKSPACE;
  const coopt_layer_io io = {cache, k_new, v_new, slot_mapping, q, out};
  DecodeCall a = attention_call(&io, 1, max_blocks_per_seq, batch, num_q_heads, chunk_size, sm_scale, workspace);
  a.plan = plan;
  a.kv_token_stride = kv_token_stride;
  if ((flags & COOPT_FLAG_OVERLAP_PREVIOUS) != 0) a.order = kOverlapPrevious;
  return launch_decode(a, static_cast<cudaStream_t>(stream));
}

int coopt_decode_layers(const coopt_layer_io* layers, int32_t num_layers, int64_t kv_token_stride, const int32_t* block_table,
                        int32_t max_blocks_per_seq, const int32_t* context_lens, int32_t batch, int32_t num_q_heads,
                        float sm_scale, void* plan, size_t plan_bytes_given, void* workspace, size_t workspace_bytes,
                        uint32_t flags, void* stream) {
  if (!layers || num_layers <= 0) return COOPT_ERR_INVALID_ARG;
  // every check of every layer before anything is launched
  const coopt_cache* c0 = layers[0].cache;
  for (int32_t l = 0; l < num_layers; ++l) {
    const coopt_layer_io& io = layers[l];
    const int rc = check_attention_shapes(io.cache, io.q, io.out, max_blocks_per_seq, batch, num_q_heads);
    if (rc != COOPT_OK) return rc;
    if (!is_fp8(io.cache->dtype) || io.cache->dtype != c0->dtype) return COOPT_ERR_UNSUPPORTED;
    if (io.cache->num_kv_heads != c0->num_kv_heads || io.cache->head_dim != c0->head_dim || io.cache->num_blocks != c0->num_blocks)
      return COOPT_ERR_INVALID_ARG;                                             // one plan serves every layer
    const bool append = io.k_new || io.v_new || io.slot_mapping;
    if (append && (!io.k_new || !io.v_new || !io.slot_mapping || kv_token_stride < static_cast<int64_t>(c0->num_kv_heads) * c0->head_dim))
      return COOPT_ERR_INVALID_ARG;
  }
  int rc = check_plan_args(batch, c0->num_kv_heads, max_blocks_per_seq, 0, plan, plan_bytes_given);
  if (rc != COOPT_OK) return rc;
  if (!block_table || !context_lens) return COOPT_ERR_INVALID_ARG;
  if ((flags & ~static_cast<uint32_t>(COOPT_FLAG_OVERLAP_PREVIOUS)) != 0) return COOPT_ERR_INVALID_ARG;
  if (batch == 0) return COOPT_OK;
  if (!workspace || workspace_bytes < workspace_need(batch, num_q_heads, c0->num_kv_heads, c0->head_dim, max_blocks_per_seq, 0, 1))
    return COOPT_ERR_WORKSPACE;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  rc = launch_decode_plan(block_table, max_blocks_per_seq, context_lens, batch, c0->num_kv_heads, c0->num_blocks, 0, plan, st);
  for (int32_t l = 0; l < num_layers && rc == COOPT_OK;) {
    const LayersLaunch next = next_layers(layers + l, num_layers - l, l == 0, kv_token_stride, block_table, max_blocks_per_seq, context_lens, batch,
                                          num_q_heads, workspace_bytes, (flags & COOPT_FLAG_OVERLAP_PREVIOUS) != 0);
    DecodeCall a = attention_call(layers + l, next.layers, max_blocks_per_seq, batch, num_q_heads, 0, sm_scale, workspace);
    a.kv_token_stride = kv_token_stride;
    if (next.early) a.order = kOverlapPrevious;
    if (l == 0 && next.early) {
      // behind the planning kernel, which copies lengths and table: this launch reads them where it read them
      a.block_table = block_table;
      a.context_lens = context_lens;
    } else {
      a.plan = plan;                     // (early: the layers before may still drain while this launch reads the plan and its own caches)
    }
    rc = launch_decode(a, st);
    l += next.layers;
  }
  return rc;
}

int coopt_selftest_layers_launch(const coopt_layer_io* layers, int32_t num_layers, int64_t kv_token_stride, const int32_t* block_table,
                                 int32_t max_blocks_per_seq, const int32_t* context_lens, int32_t batch, int32_t num_q_heads,
                                 size_t workspace_bytes, uint32_t flags, int32_t* layers_of_launch, int32_t* early) {
  if (!layers || num_layers <= 0 || !layers_of_launch || !early) return COOPT_ERR_INVALID_ARG;
  for (int32_t l = 0; l < num_layers;) {
    const LayersLaunch next = next_layers(layers + l, num_layers - l, l == 0, kv_token_stride, block_table, max_blocks_per_seq, context_lens, batch,
                                          num_q_heads, workspace_bytes, (flags & COOPT_FLAG_OVERLAP_PREVIOUS) != 0);
    for (int32_t k = 0; k < next.layers; ++k, ++l) {
      layers_of_launch[l] = next.layers;
      early[l] = next.early ? 1 : 0;
    }
  }
  return COOPT_OK;
}

int coopt_paged_chunked(const coopt_cache* cache, const void* q, void* out, const int32_t* cu_q_lens,
                        const int32_t* block_table, int32_t max_blocks_per_seq, const int32_t* context_lens,
                        int32_t batch, int32_t num_q_heads, int32_t total_q, int32_t chunk_size, int32_t causal,
                        float sm_scale, void* workspace, size_t workspace_bytes, void* stream) {
  const int rc = check_attention_args(cache, q, out, block_table, max_blocks_per_seq, context_lens, batch, num_q_heads);
  if (rc != COOPT_OK) return rc;
  if (!cu_q_lens || total_q < batch) return COOPT_ERR_INVALID_ARG;
  if (chunk_size <= 0 || chunk_size % kBlockSize != 0 || chunk_size / kBlockSize > decode_max_chunk_blocks())
    return COOPT_ERR_INVALID_ARG;
  if (batch == 0) return COOPT_OK;
  if (!workspace || workspace_bytes < workspace_need(batch, num_q_heads, cache->num_kv_heads, cache->head_dim, max_blocks_per_seq, chunk_size, 1))
    return COOPT_ERR_WORKSPACE;
  if (total_q == batch) {
    // one query token per sequence: the Opt-Pa chunk-and-merge decode
    const coopt_layer_io io = {cache, nullptr, nullptr, nullptr, q, out};
    DecodeCall a = attention_call(&io, 1, max_blocks_per_seq, batch, num_q_heads, chunk_size, sm_scale, workspace);
    a.block_table = block_table;
    a.context_lens = context_lens;
    a.cu_q_lens = cu_q_lens;
    return launch_decode(a, static_cast<cudaStream_t>(stream));
  }
  return launch_paged_prefill(cache, q, out, cu_q_lens, block_table, max_blocks_per_seq, context_lens, batch,
                              num_q_heads, total_q, causal, sm_scale, workspace, num_sms(), static_cast<cudaStream_t>(stream));
}

namespace {
// The device's address of a host pointer if the memory is page-locked and mapped (cudaHostAlloc, cudaHostRegister),
// null for pageable memory (and for anything that is not host memory).
const uint8_t* mapped_host_pointer(const void* host) {
  cudaPointerAttributes attr;
  if (cudaPointerGetAttributes(&attr, host) != cudaSuccess) {
    (void)cudaGetLastError();
    return nullptr;
  }
  if (attr.type != cudaMemoryTypeHost || attr.devicePointer == nullptr) return nullptr;
  return static_cast<const uint8_t*>(attr.devicePointer);
}

coopt_step_layout step_layout(int batch, int hq, int hkv, int d, int max_blocks) {
  auto up = [](size_t x) { return (x + 255) / 256 * 256; };
  coopt_step_layout s;
  size_t at = 0;
  s.q = at;            at += up(static_cast<size_t>(batch) * hq * d * 2);
  s.k_new = at;        at += up(static_cast<size_t>(batch) * hkv * d * 2);
  s.v_new = at;        at += up(static_cast<size_t>(batch) * hkv * d * 2);
  s.slot_mapping = at; at += up(static_cast<size_t>(batch) * 8);
  s.block_table = at;  at += up(static_cast<size_t>(batch) * max_blocks * 4);
  s.context_lens = at; at += up(static_cast<size_t>(batch) * 4);
  s.in_bytes = at;
  s.out = at;          at += up(static_cast<size_t>(batch) * hq * d * 2);
  s.out_bytes = static_cast<size_t>(batch) * hq * d * 2;
  s.total_bytes = at;
  return s;
}
}  // namespace

int coopt_step_staging_layout(int32_t batch, int32_t num_q_heads, int32_t num_kv_heads, int32_t head_dim,
                              int32_t max_blocks_per_seq, coopt_step_layout* layout) {
  if (batch < 0 || num_q_heads <= 0 || num_kv_heads <= 0 || head_dim <= 0 || max_blocks_per_seq <= 0 || !layout) return COOPT_ERR_INVALID_ARG;
  *layout = step_layout(batch, num_q_heads, num_kv_heads, head_dim, max_blocks_per_seq);
  return COOPT_OK;
}

int coopt_decode_step_host(const coopt_cache* cache, const void* step_inputs_host, void* out_host, int32_t max_blocks_per_seq,
                           int32_t batch, int32_t num_q_heads, float sm_scale, void* staging, size_t staging_bytes, void* plan,
                           size_t plan_bytes_given, void* workspace, size_t workspace_bytes, void* stream) {
  int rc = check_cache(cache);
  if (rc != COOPT_OK) return rc;
  if (!step_inputs_host || !out_host || batch < 0 || num_q_heads <= 0 || max_blocks_per_seq <= 0) return COOPT_ERR_INVALID_ARG;
  if (batch == 0) return COOPT_OK;
  const int hkv = cache->num_kv_heads, d = cache->head_dim;
  const coopt_step_layout s = step_layout(batch, num_q_heads, hkv, d, max_blocks_per_seq);
  if (!staging || staging_bytes < s.total_bytes) return COOPT_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(staging) % 256 != 0) return COOPT_ERR_INVALID_ARG;
  uint8_t* dev = static_cast<uint8_t*>(staging);
  // every check of the device part before the first copy is enqueued
  rc = check_attention_args(cache, dev + s.q, dev + s.out, reinterpret_cast<const int32_t*>(dev + s.block_table), max_blocks_per_seq,
                            reinterpret_cast<const int32_t*>(dev + s.context_lens), batch, num_q_heads);
  if (rc != COOPT_OK) return rc;
  if (!is_fp8(cache->dtype)) return COOPT_ERR_UNSUPPORTED;
  rc = check_plan_args(batch, hkv, max_blocks_per_seq, 0, plan, plan_bytes_given);
  if (rc != COOPT_OK) return rc;
  if (!workspace || workspace_bytes < workspace_need(batch, num_q_heads, hkv, d, max_blocks_per_seq, 0, 1)) return COOPT_ERR_WORKSPACE;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  coopt_layer_io io = {cache, dev + s.k_new, dev + s.v_new, reinterpret_cast<const int64_t*>(dev + s.slot_mapping), dev + s.q, dev + s.out};
  DecodeCall a = attention_call(&io, 1, max_blocks_per_seq, batch, num_q_heads, 0, sm_scale, workspace);
  a.plan = plan;
  a.kv_token_stride = static_cast<int64_t>(hkv) * d;
  // Host buffers that are page-locked and mapped into the device's address space are used where they are: the
  // kernel fetches the queries and the new tokens from them and stores the result into them, and only the
  // index arrays (slots, block table, context lengths: what the planner walks) are copied to the device.
  const uint8_t* in_dev = mapped_host_pointer(step_inputs_host);
  uint8_t* out_dev = const_cast<uint8_t*>(mapped_host_pointer(out_host));
  const bool in_place = in_dev != nullptr && out_dev != nullptr && reinterpret_cast<uintptr_t>(in_dev) % 16 == 0 && reinterpret_cast<uintptr_t>(out_dev) % 16 == 0;
  const size_t from = in_place ? s.slot_mapping : 0;
  if (cudaMemcpyAsync(dev + from, static_cast<const uint8_t*>(step_inputs_host) + from, s.in_bytes - from, cudaMemcpyHostToDevice, st) != cudaSuccess)
    return COOPT_ERR_CUDA;
  rc = launch_decode_plan(reinterpret_cast<const int32_t*>(dev + s.block_table), max_blocks_per_seq,
                          reinterpret_cast<const int32_t*>(dev + s.context_lens), batch, hkv, cache->num_blocks, 0, plan, st);
  if (rc != COOPT_OK) return rc;
  if (in_place) {
    io.q = in_dev + s.q; io.k_new = in_dev + s.k_new; io.v_new = in_dev + s.v_new; io.out = out_dev;
    return launch_decode(a, st);
  }
  rc = launch_decode(a, st);
  if (rc != COOPT_OK) return rc;
  return cudaMemcpyAsync(out_host, dev + s.out, s.out_bytes, cudaMemcpyDeviceToHost, st) == cudaSuccess ? COOPT_OK : COOPT_ERR_CUDA;
}

const char* coopt_status_string(int status) {
  switch (status) {
    case COOPT_OK: return "ok";
    case COOPT_ERR_INVALID_ARG: return "invalid argument";
    case COOPT_ERR_UNSUPPORTED: return "unsupported shape";
    case COOPT_ERR_WORKSPACE: return "workspace missing or too small";
    case COOPT_ERR_CUDA: return "CUDA runtime error";
    case COOPT_ERR_TIMEOUT: return "device-side wait timed out";
    default: return "unknown status";
  }
}

int coopt_version(void) { return 200; }

}  // extern "C"
