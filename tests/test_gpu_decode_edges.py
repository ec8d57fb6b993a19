"""GPU parity of the decode kernel where its work decomposition can go wrong: lengths around block edges, units that
warps and CTAs share or take whole, full batches of the shortest contexts, group sizes 1 and 8, every cache format."""
import numpy as np
import pytest
import torch

from oracle import attention, e5m2, kv_cache
from paper_2602_09323_b200 import binding, workloads
from tests import helpers

pytestmark = pytest.mark.gpu

CASES = {
    "one token": [1],
    "block edges": [15, 16, 17, 31, 32, 33, 0, 1],
    "whole units and cut ones": [511, 512, 513, 1024, 1025, 3072, 3073],
    "a full batch of the shortest": [1 + (7 * i) % 40 for i in range(512)],
    "one long among empty ones": [0, 0, 9000, 0],
    "more places than fit one share": [700 + 13 * i for i in range(40)],
}


@pytest.mark.parametrize("case", list(CASES))
@pytest.mark.parametrize("hq,hkv,d,fmt", [(8, 1, 128, "e4m3"), (2, 2, 64, "e5m2"), (12, 4, 64, "e4m3"), (7, 1, 128, "bf16"), (5, 1, 128, "e5m2")])
def test_shares_of_the_line(case, hq, hkv, d, fmt):
    """Tolerance: the repository's bound for every decode path (helpers.check_attention: bf16 output rounding plus
    probabilities of 11 bits)."""
    w = workloads.make_workload("edges", CASES[case], hq, hkv, d, seed=hq + d)
    if fmt == "bf16":
        cache = helpers.gpu_fill(w, dtype=binding.KV_BF16)
        kv = kv_cache.new_cache_bf16(w.num_blocks, hkv, d)
        kv_cache.kv_write_bf16(kv, w.k.float().numpy(), w.v.float().numpy(), w.slot_mapping.numpy())
    elif fmt == "e5m2":
        cache = helpers.gpu_fill(w, dtype=binding.KV_FP8_E5M2)
        kv = (*helpers.oracle_fp8_cache(w, fmt=e5m2), e5m2)
    else:
        cache = helpers.gpu_fill(w)
        kv = helpers.oracle_fp8_cache(w)
    ref = attention.paged_attention(w.q.float().numpy(), kv, w.block_table.numpy(), w.context_lens)
    out, ws = helpers.gpu_decode(w, cache)
    helpers.check_attention(out, ref, what=f"{case} {fmt}")
    again = binding.paged_decode(cache, w.q.cuda(), w.block_table.cuda(), w.context_lens_tensor.cuda(), w.sm_scale, ws)
    assert torch.equal(out, again)                      # the piece counters were left ready, and the merge order is fixed


@pytest.mark.parametrize("chunk", [16, 48, 512])
@pytest.mark.parametrize("case", ["block edges", "whole units and cut ones", "one long among empty ones"])
def test_chunks_that_warps_and_ctas_share(case, chunk):
    w = workloads.make_workload("edges", CASES[case], 6, 2, 128, seed=chunk)
    out, ws = helpers.gpu_decode(w, helpers.gpu_fill(w), chunk_size=chunk)
    ref, partials = attention.paged_attention_chunked(w.q.float().numpy(), helpers.oracle_fp8_cache(w), w.block_table.numpy(), w.context_lens, chunk)
    helpers.check_attention(out, ref, what=f"{case} chunk {chunk}")
    o_c, m_c, l_c = (t.cpu().numpy() for t in binding.chunk_partials(ws, w.batch, 6, 128, w.block_table.shape[1], chunk))
    for (b, h), (m, l, o) in partials.items():          # bounds of tests/test_gpu_decode.py: f16 probabilities, fp32 sums
        n = len(m)
        assert np.allclose(m_c[b, h, :n], m, rtol=1e-4, atol=1e-3)
        assert np.allclose(l_c[b, h, :n], l, rtol=5e-3, atol=1e-4)
        assert np.allclose(o_c[b, h, :n], o, rtol=5e-3, atol=2e-2)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("lens,hkv,chunk", [([0, 0, 9000], 2, 512), ([9000, 0, 0, 9000, 1], 2, 512), ([0, 0, 9000, 0], 2, 512),
                                            ([0, 0, 131072, 131072], 1, 2048)])
def test_chunks_longer_than_a_share_beside_empty_contexts(lens, hkv, chunk, d):
    """The longest chunk counts whatever else is empty: every row is stored, and no piece is left counted for a later call."""
    w = workloads.make_workload("empties", lens, 2 * hkv, hkv, d, seed=d)
    cache, kv = helpers.gpu_fill(w), helpers.oracle_fp8_cache(w)
    ws = binding.new_workspace(w.batch, 2 * hkv, hkv, d, w.block_table.shape[1], chunk, w.batch)
    for now in (lens, [L * 3 // 5 for L in lens]):
        out = torch.full(w.q.shape, float("nan"), dtype=torch.bfloat16, device="cuda")
        binding.paged_chunked(cache, w.q.cuda(), w.cu_q_lens.cuda(), w.block_table.cuda(), torch.tensor(now, dtype=torch.int32).cuda(), chunk, True, w.sm_scale, ws, out=out)
        torch.cuda.synchronize()
        assert binding.workspace_status(ws) == 0
        assert not ws[256:256 + 4 * 16384].any(), "piece counters"
        ref, _ = attention.paged_attention_chunked(w.q.float().numpy(), kv, w.block_table.numpy(), now, chunk)
        helpers.check_attention(out, ref, what=f"{now} chunk {chunk}")


@pytest.mark.parametrize("hq,hkv,d,lens", [(8, 2, 128, [300, 1, 0, 17, 2048]), (16, 2, 64, [16, 33, 1, 900])])
@pytest.mark.parametrize("n,how", [(2, "apart"), (3, "chained"), (3, "some append"), (67, "apart"), (2, "one output")])
def test_layers_in_one_launch_equal_layers_one_by_one(hq, hkv, d, lens, n, how):
    """Layers whose buffers are apart share a launch; layers that read what another writes must still run in order
    ("chained": a layer's output is the next one's query; "one output": the last layer's result stays)."""
    w = workloads.make_workload("layers", lens, hq, hkv, d, seed=n)
    table, lens_t, B, gen = w.block_table.cuda(), w.context_lens_tensor.cuda(), w.batch, torch.Generator("cuda").manual_seed(n)
    draw = lambda heads: torch.randn(B, heads, d, generator=gen, device="cuda").to(torch.bfloat16)
    live = torch.tensor([L > 0 for L in lens], device="cuda")
    at = torch.tensor([w.kv_offsets[b] + max(L, 1) - 1 for b, L in enumerate(lens)]).clamp(max=w.k.shape[0] - 1)
    slots = torch.where(live, w.slot_mapping[at].cuda(), torch.full((B,), -1, device="cuda"))
    hist = np.concatenate([np.arange(w.kv_offsets[b], w.kv_offsets[b] + max(0, L - 1)) for b, L in enumerate(lens)])
    base = helpers.gpu_fill(w, calls=[hist])
    qs, outs = [draw(hq) for _ in range(n)], [torch.full((B, hq, d), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(n)]
    if how == "chained":
        qs[1:] = outs[:-1]
    if how == "one output":
        outs = [outs[0]] * n
    new = [(draw(hkv), draw(hkv), slots) if how != "some append" or y % 2 else (None, None, None) for y in range(n)]

    def run(together):
        caches = []
        for _ in range(n):
            c = binding.Cache(w.num_blocks, hkv, d)
            c.data.copy_(base.data)
            caches.append(c)
        ws = binding.new_workspace(B, hq, hkv, d, table.shape[1])
        if together:
            plan = torch.empty(binding.plan_bytes(B, hkv, table.shape[1]), dtype=torch.uint8, device="cuda")
            ios = [{"cache": c, "q": q, "out": o, "k_new": k, "v_new": v, "slot_mapping": s} for c, q, o, (k, v, s) in zip(caches, qs, outs, new)]
            layer_set = binding.LayerSet(ios)
            layer_set.kv_stride = hkv * d
            binding.decode_layers(layer_set, table, lens_t, hq, w.sm_scale, plan, ws)
            # the plan is one that a later launch can use
            again = binding.decode_step_planned(caches[0], plan, qs[0], table.shape[1], w.sm_scale, ws)
            assert how != "apart" or torch.equal(again, outs[0])
        else:
            for c, q, o, (k, v, s) in zip(caches, qs, outs, new):
                if k is not None:
                    binding.kv_write(c, k, v, s)
                binding.paged_decode(c, q, table, lens_t, w.sm_scale, ws, out=o)
        torch.cuda.synchronize()
        assert binding.workspace_status(ws) == 0
        return [o.clone() for o in outs], [c.data for c in caches]

    (want, want_bytes), (got, got_bytes) = run(False), run(True)
    for y in range(n):
        assert torch.equal(want_bytes[y], got_bytes[y]), f"layer {y}: cache bytes"
        assert torch.equal(got[y], want[y]), f"layer {y}: outputs"


@pytest.mark.parametrize("lens", [[64, 0, 1, 49, 16], [1 + i % 64 for i in range(300)], [65, 3, 64], [1 + 7 * i % 192 for i in range(288)],
                                  [1 + 7 * i % 193 for i in range(193)]])
@pytest.mark.parametrize("hq,hkv,d,n", [(8, 8, 128, 8), (10, 2, 64, 3)])
def test_layers_of_units_around_the_most_that_a_warp_holds_whole(hq, hkv, d, n, lens):
    test_layers_in_one_launch_equal_layers_one_by_one(hq, hkv, d, lens, n, "apart")


@pytest.mark.parametrize("lens", [[70, 300, 900, 3072], [80, 176, 3073], [70, 0, 300], [200] * 74])
@pytest.mark.parametrize("d,n", [(128, 5), (64, 2)])
def test_layers_whose_shares_are_their_units(d, n, lens):
    """On both sides of the longest unit that is held whole, with an empty context, and with as many units as there are CTAs."""
    test_layers_in_one_launch_equal_layers_one_by_one(6, 2, d, lens, n, "apart")


@pytest.mark.parametrize("hq,hkv,d", [(16, 2, 128), (10, 2, 64)])
def test_pieces_of_many_rounds_are_read_behind_their_writers(hq, hkv, d):
    """Eight layers a launch whose units are cut between all warps and CTAs, again and again: the same bits every time."""
    for _ in range(4):
        test_layers_in_one_launch_equal_layers_one_by_one(hq, hkv, d, [1500 + 61 * i for i in range(16)], 8, "apart")


def _tiny_values(lens, fmt, d, spans):
    """A workload without outlier channels whose V is N(0, 1) times 2^-124 (a block's scale is then below 2^-128, whose
    reciprocal is not a number of 32 bits) at the positions ``spans`` of every sequence."""
    w = workloads.make_workload("tiny", lens, 6, 2, d, seed=d + len(lens), outliers=False)
    for b, L in enumerate(lens):
        for lo, hi in spans:
            rows = slice(w.kv_offsets[b] + min(lo, L), w.kv_offsets[b] + min(hi, L))
            w.v[rows] = (w.v[rows].float() * 2.0 ** -124).to(torch.bfloat16)
    kv = helpers.oracle_fp8_cache(w) if fmt == "e4m3" else (*helpers.oracle_fp8_cache(w, fmt=e5m2), e5m2)
    return w, helpers.gpu_fill(w, dtype=binding.KV_FP8_E4M3 if fmt == "e4m3" else binding.KV_FP8_E5M2), kv


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("fmt", ["e4m3", "e5m2"])
@pytest.mark.parametrize("lens", [[40, 16, 700, 3000], [9, 64, 33] * 40])
def test_v_scales_whose_reciprocal_overflows(lens, fmt, d):
    """Tiny blocks in front of, between and behind ordinary ones count for nothing beside them, and alone they keep their
    values: bf16 rounding (2^-9 of the result, or half of 2^-133 among subnormals) plus 11 bits of probabilities."""
    w, cache, kv = _tiny_values(lens, fmt, d, [(0, 32), (64, 80), (1500, 2000)])
    ref = attention.paged_attention(w.q.float().numpy(), kv, w.block_table.numpy(), w.context_lens)
    out, _ = helpers.gpu_decode(w, cache)
    helpers.check_attention(out, ref, what=f"tiny blocks {fmt}")
    helpers.check_attention(helpers.gpu_decode(w, cache, chunk_size=32)[0], ref, what=f"tiny blocks in chunks {fmt}")
    w, cache, kv = _tiny_values(lens, fmt, d, [(0, 1 << 20)])
    ref = attention.paged_attention(w.q.float().numpy(), kv, w.block_table.numpy(), w.context_lens)
    got = helpers.gpu_decode(w, cache)[0].double().cpu().numpy()
    bound = 2.0 ** -8 * np.abs(ref) + 2.0 ** -134 + 2.0 ** -11 * float(w.v.float().abs().max())
    assert np.all(np.abs(got - ref) <= bound), np.max(np.abs(got - ref) / bound)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("lens", [[640], [641], [640, 0, 300], [639, 657]])
def test_bf16_units_around_the_longest_that_are_not_cut(lens, d):
    w = workloads.make_workload("bf16", lens, 6, 2, d, seed=lens[0])
    kv = kv_cache.new_cache_bf16(w.num_blocks, 2, d)
    kv_cache.kv_write_bf16(kv, w.k.float().numpy(), w.v.float().numpy(), w.slot_mapping.numpy())
    out, _ = helpers.gpu_decode(w, helpers.gpu_fill(w, dtype=binding.KV_BF16))
    helpers.check_attention(out, attention.paged_attention(w.q.float().numpy(), kv, w.block_table.numpy(), w.context_lens), what=f"bf16 {lens}")


@pytest.mark.parametrize("d,fmt", [(64, "e4m3"), (128, "e4m3"), (64, "bf16"), (128, "bf16")])
@pytest.mark.parametrize("chunk", [512, 2048, 32768])
def test_a_context_in_a_single_chunk_beside_longer_ones(chunk, d, fmt):
    """Whole in a warp, shared by warps, shared by CTAs: output and exported partials."""
    w = workloads.make_workload("one chunk", [9000, 1, 512, 513, 0, 2048, 30, 2049], 6, 2, d, seed=chunk + d)
    if fmt == "bf16":
        kv = kv_cache.new_cache_bf16(w.num_blocks, 2, d)
        kv_cache.kv_write_bf16(kv, w.k.float().numpy(), w.v.float().numpy(), w.slot_mapping.numpy())
    else:
        kv = helpers.oracle_fp8_cache(w)
    out, ws = helpers.gpu_decode(w, helpers.gpu_fill(w, dtype=binding.KV_BF16 if fmt == "bf16" else binding.KV_FP8_E4M3), chunk_size=chunk)
    ref, partials = attention.paged_attention_chunked(w.q.float().numpy(), kv, w.block_table.numpy(), w.context_lens, chunk)
    helpers.check_attention(out, ref, what=f"chunk {chunk} {fmt}")
    o_c, m_c, l_c = (t.cpu().numpy() for t in binding.chunk_partials(ws, w.batch, 6, d, w.block_table.shape[1], chunk))
    for (b, h), (m, l, o) in partials.items():          # bounds as above
        n = len(m)
        assert np.allclose(m_c[b, h, :n], m, rtol=1e-4, atol=1e-3)
        assert np.allclose(l_c[b, h, :n], l, rtol=5e-3, atol=1e-4)
        assert np.allclose(o_c[b, h, :n], o, rtol=5e-3, atol=2e-2)


def test_views_with_a_further_dimension_are_taken_as_before():
    w = workloads.make_workload("views", [40, 17], 4, 2, 64, seed=5)
    plain, cache = helpers.gpu_fill(w), binding.Cache(w.num_blocks, 2, 64)
    binding.kv_write(cache, w.k.cuda()[..., None], w.v.cuda()[..., None], w.slot_mapping.cuda())
    assert torch.equal(cache.data, plain.data)
    out, ws = helpers.gpu_decode(w, cache)
    q = w.q.cuda().view(w.batch, 4, 2, 32)
    again = binding.paged_decode(cache, q, w.block_table.cuda(), w.context_lens_tensor.cuda(), w.sm_scale, ws)
    assert again.shape == q.shape and torch.equal(again.view_as(out), out)


@pytest.mark.parametrize("fmt", ["e4m3", "e5m2"])
@pytest.mark.parametrize("d", [64, 128])
def test_codes_past_the_context_do_not_count(d, fmt):
    """Contexts that end anywhere in a block, the first or a later one, with codes that are no numbers in all slots past the end.  The result is that of a clean cache, bit for bit
    (a slot past the end counts for nothing), and the cache is left as it is."""
    lens = [1, 5, 16, 17, 31, 32, 33, 47, 48, 63, 700, 2049]
    kind = {"e4m3": binding.KV_FP8_E4M3, "e5m2": binding.KV_FP8_E5M2}[fmt]
    w = workloads.make_workload("past the end", lens, 6, 2, d, seed=d)
    cache = helpers.gpu_fill(w, dtype=kind)
    out, ws = helpers.gpu_decode(w, cache)
    kv = (*helpers.oracle_fp8_cache(w, fmt=e5m2), e5m2) if fmt == "e5m2" else helpers.oracle_fp8_cache(w)
    helpers.check_attention(out, attention.paged_attention(w.q.float().numpy(), kv, w.block_table.numpy(), w.context_lens), what=f"past the end {fmt}")
    at = [binding.cache_offset(cache, int(w.block_table[b, (L - 1) // 16]), g, which, t, e)
          for b, L in enumerate(lens) for g in range(2) for which in (0, 1) for t in range((L - 1) % 16 + 1, 16) for e in range(d)]
    cache.data[torch.tensor(at, device="cuda")] = 0x7F
    before = cache.data.clone()
    table, lens_t = w.block_table.cuda(), w.context_lens_tensor.cuda()
    assert torch.equal(binding.paged_decode(cache, w.q.cuda(), table, lens_t, w.sm_scale, ws), out)
    outs = [torch.full_like(out, float("nan")) for _ in range(3)]          # layers in one launch
    layers = binding.LayerSet([{"cache": cache, "q": w.q.cuda(), "out": o} for o in outs])
    plan = torch.empty(binding.plan_bytes(w.batch, 2, table.shape[1]), dtype=torch.uint8, device="cuda")
    binding.decode_layers(layers, table, lens_t, 6, w.sm_scale, plan, ws)
    assert all(torch.equal(o, out) for o in outs)
    assert torch.equal(cache.data, before)


@pytest.mark.parametrize("loud", ["V scale", "logits"])
@pytest.mark.parametrize("fmt", ["e4m3", "e5m2"])
@pytest.mark.parametrize("d", [64, 128])
def test_a_block_keeps_its_bits_beside_one_that_dwarfs_it(d, fmt, loud):
    """The last block of a context moves a reference by 2^20 to 2^40, and all of its V but one value is zero: the other dims'
    results are those of the blocks in front of it.  V is not negative there, so every product is in the sum with its own sign,
    and the result is off by no more than its terms are, 2^-11 (a probability of 11 bits, rounded to nearest: 2^-12, and less than
    that again for fp32 exponentials and sums), and by the rounding of the bf16 result, of 8 bits, to nearest: 2^-8 at most."""
    lens, bits = [32, 29, 17, 64, 61, 32, 32], [20, 24, 28, 32, 36, 40, 30]
    w = workloads.make_workload("dwarfed", lens, 6, 2, d, seed=d, outliers=False)
    w.v.copy_(w.v.abs())
    w.q.fill_(1.0)
    w.k.mul_(0.125)
    for b, (L, e) in enumerate(zip(lens, bits)):
        rows = slice(w.kv_offsets[b] + (L - 1) // 16 * 16, w.kv_offsets[b] + L)      # the last block, the second or the fourth
        w.v[rows] = 0
        if loud == "V scale":
            w.v[w.kv_offsets[b] + L - 1, :, 0] = 2.0 ** e
        else:
            w.k[rows] = e * np.log(2.0) / np.sqrt(d)
    kind = binding.KV_FP8_E4M3 if fmt == "e4m3" else binding.KV_FP8_E5M2
    kv = helpers.oracle_fp8_cache(w) if fmt == "e4m3" else (*helpers.oracle_fp8_cache(w, fmt=e5m2), e5m2)
    ref = attention.paged_attention(w.q.float().numpy(), kv, w.block_table.numpy(), w.context_lens)[..., 1:]
    cache = helpers.gpu_fill(w, dtype=kind)
    out, ws = helpers.gpu_decode(w, cache)
    outs = [torch.full_like(out, float("nan")) for _ in range(2)]          # layers in one launch
    layers = binding.LayerSet([{"cache": cache, "q": w.q.cuda(), "out": o} for o in outs])
    plan = torch.empty(binding.plan_bytes(w.batch, 2, w.block_table.shape[1]), dtype=torch.uint8, device="cuda")
    binding.decode_layers(layers, w.block_table.cuda(), w.context_lens_tensor.cuda(), 6, w.sm_scale, plan, ws)
    assert torch.equal(outs[0], out) and torch.equal(outs[1], out)
    chunked = helpers.gpu_decode(w, cache, chunk_size=32)[0]
    for got in (out, chunked):
        off = np.abs(got.double().cpu().numpy()[..., 1:] - ref)
        assert np.all(off <= (2.0 ** -8 + 2.0 ** -11) * ref), np.max(off / ref)


@pytest.mark.parametrize("d", [64, 128])
def test_an_infinite_value_is_an_infinite_result(d):
    """An E5M2 cache that comes from elsewhere may hold infinities (the write saturates).  One in V at a valid token makes its
    dim's result infinite and no other, wherever the context ends behind it, for one layer and for several in a launch."""
    lens = [1, 5, 16, 17, 20, 32, 33, 48, 80, 700]
    w = workloads.make_workload("infinite", lens, 6, 2, d, seed=d, outliers=False)
    w.q.mul_(0.25)                                                         # every probability is an f16 number
    cache = helpers.gpu_fill(w, dtype=binding.KV_FP8_E5M2)
    clean, ws = helpers.gpu_decode(w, cache)
    at = [binding.cache_offset(cache, int(w.block_table[b, (L - 1) // 16]), g, 1, (L - 1) % 16, 3 + g) for b, L in enumerate(lens) for g in range(2)]
    cache.data[torch.tensor(at, device="cuda")] = torch.tensor([0x7C, 0xFC] * len(lens), dtype=torch.uint8, device="cuda")
    want = clean.clone()
    want[:, :3, 3], want[:, 3:, 4] = float("inf"), float("-inf")
    table, lens_t = w.block_table.cuda(), w.context_lens_tensor.cuda()
    assert torch.equal(binding.paged_decode(cache, w.q.cuda(), table, lens_t, w.sm_scale, ws), want)
    outs = [torch.full_like(clean, float("nan")) for _ in range(2)]        # layers in one launch
    layers = binding.LayerSet([{"cache": cache, "q": w.q.cuda(), "out": o} for o in outs])
    plan = torch.empty(binding.plan_bytes(w.batch, 2, table.shape[1]), dtype=torch.uint8, device="cuda")
    binding.decode_layers(layers, table, lens_t, 6, w.sm_scale, plan, ws)
    assert torch.equal(outs[0], want) and torch.equal(outs[1], want)


@pytest.mark.parametrize("hq,hkv,d,fmt", [(64, 8, 128, "e4m3"), (16, 8, 128, "e5m2"), (64, 8, 64, "e4m3")])
def test_long_layers_in_one_launch_equal_layers_one_by_one(hq, hkv, d, fmt):
    """Three layers of 64 sequences in block tables of 128 columns, 440 blocks a multiprocessor: units cut between warps and CTAs
    in every layer, with appended tokens.  All sequences have their first 95 blocks in common, and what follows to themselves."""
    B, shared, width, n = 64, 95, 128, 3
    gen = torch.Generator("cuda").manual_seed(hq + d)
    draw = lambda *shape: torch.randn(*shape, generator=gen, device="cuda").to(torch.bfloat16)
    lens = [shared * 16 + 1 + (37 * b) % (16 * (width - shared)) for b in range(B)]
    own = width - shared
    table = torch.full((B, width), -1, dtype=torch.int32)
    for b, L in enumerate(lens):
        table[b, :shared] = torch.arange(shared)
        k = -(-L // 16) - shared
        table[b, shared:shared + k] = shared + own * b + torch.arange(k)
    blocks = shared + own * B
    table, lens_t = table.cuda(), torch.tensor(lens, dtype=torch.int32).cuda()
    last = lens_t.long() - 1
    slots = table.gather(1, (last // 16)[:, None])[:, 0].long() * 16 + last % 16
    kind = {"e4m3": binding.KV_FP8_E4M3, "e5m2": binding.KV_FP8_E5M2}[fmt]
    ws = binding.new_workspace(B, hq, hkv, d, width)
    ios, want, want_bytes = [], [], []
    for y in range(n):
        cache = binding.Cache(blocks, hkv, d, kind)
        binding.kv_write(cache, draw(blocks * 16, hkv, d), draw(blocks * 16, hkv, d), torch.arange(blocks * 16, device="cuda"))
        io = {"cache": cache, "q": draw(B, hq, d), "out": torch.full((B, hq, d), float("nan"), dtype=torch.bfloat16, device="cuda"),
              "k_new": draw(B, hkv, d), "v_new": draw(B, hkv, d), "slot_mapping": slots}
        twin = binding.Cache(blocks, hkv, d, kind)
        twin.data.copy_(cache.data)
        binding.kv_write(twin, io["k_new"], io["v_new"], slots)
        want.append(binding.paged_decode(twin, io["q"], table, lens_t, d ** -0.5, ws))
        want_bytes.append(twin.data)
        ios.append(io)
    plan = torch.empty(binding.plan_bytes(B, hkv, width), dtype=torch.uint8, device="cuda")
    for keys in (set(ios[0]), {"cache", "q", "out"}):                       # with the new tokens, and over what they have left
        layer_set = binding.LayerSet([{k: v for k, v in io.items() if k in keys} for io in ios])
        for io in ios:
            io["out"].fill_(float("nan"))
        binding.decode_layers(layer_set, table, lens_t, hq, d ** -0.5, plan, ws)
        torch.cuda.synchronize()
        assert binding.workspace_status(ws) == 0
        for y, io in enumerate(ios):
            assert torch.equal(io["out"], want[y]), f"layer {y}: outputs"
            assert torch.equal(io["cache"].data, want_bytes[y]), f"layer {y}: cache bytes"


@pytest.mark.parametrize("d", [64, 128])
def test_bf16_values_past_the_context_do_not_count(d):
    lens = [1, 5, 16, 17, 31, 33, 47, 700, 2049]
    w = workloads.make_workload("past the end", lens, 6, 2, d, seed=d)
    cache = helpers.gpu_fill(w, dtype=binding.KV_BF16)
    out, ws = helpers.gpu_decode(w, cache)
    raw = cache.data.view(torch.int16)
    at = [binding.cache_offset(cache, int(w.block_table[b, (L - 1) // 16]), g, which, t, e) // 2
          for b, L in enumerate(lens) for g in range(2) for which in (0, 1) for t in range((L - 1) % 16 + 1, 16) for e in range(d)]
    raw[torch.tensor(at, device="cuda")] = 0x7FC0                           # no number
    assert torch.equal(binding.paged_decode(cache, w.q.cuda(), w.block_table.cuda(), w.context_lens_tensor.cuda(), w.sm_scale, ws), out)
    assert torch.equal(helpers.gpu_decode(w, cache, chunk_size=512)[0][:7], out[:7])      # contexts of a single chunk


@pytest.mark.parametrize("fmt", ["e4m3", "e5m2"])
@pytest.mark.parametrize("d", [64, 128])
def test_a_token_appended_in_front_of_codes_that_are_no_numbers(d, fmt):
    """The one-launch step adds a token to a block whose later slots hold codes that are no numbers: output and cache bytes
    are those of the write followed by the decode, the later slots' codes among them."""
    lens = [2, 5, 16, 18, 31, 33, 47, 50, 63, 700, 2049]                   # (2049: the token begins its block, which is cleared)
    kind = {"e4m3": binding.KV_FP8_E4M3, "e5m2": binding.KV_FP8_E5M2}[fmt]
    w = workloads.make_workload("append in front", lens, 6, 2, d, seed=d)
    hist = np.concatenate([np.arange(w.kv_offsets[b], w.kv_offsets[b] + L - 1) for b, L in enumerate(lens)])
    new = torch.tensor([w.kv_offsets[b] + L - 1 for b, L in enumerate(lens)])
    # K and V that are small next to the block's scale, so that the write leaves the scale and the other codes as they are
    k_new, v_new, slots = (w.k[new] * 0.01).cuda(), (w.v[new] * 0.01).cuda(), w.slot_mapping[new].cuda()
    table, lens_t = w.block_table.cuda(), w.context_lens_tensor.cuda()
    caches = [helpers.gpu_fill(w, dtype=kind, calls=[hist]) for _ in range(3)]
    at = [binding.cache_offset(caches[0], int(w.block_table[b, (L - 1) // 16]), g, which, t, e)
          for b, L in enumerate(lens) for g in range(2) for which in (0, 1) for t in range((L - 1) % 16 + 1, 16) for e in range(d)]
    for c in caches:
        c.data[torch.tensor(at, device="cuda")] = 0x7F
    ws = binding.new_workspace(w.batch, 6, 2, d, table.shape[1])
    binding.kv_write(caches[0], k_new, v_new, slots)
    want = binding.paged_decode(caches[0], w.q.cuda(), table, lens_t, w.sm_scale, ws)
    assert torch.isfinite(want.float()).all()
    plan = binding.decode_plan(table, lens_t, 2, w.num_blocks)
    got = binding.decode_step_planned(caches[1], plan, w.q.cuda(), table.shape[1], w.sm_scale, ws, k_new, v_new, slots)
    assert torch.equal(got, want) and torch.equal(caches[1].data, caches[0].data)
    outs = [torch.full_like(want, float("nan")) for _ in range(2)]         # two layers in one launch, one of which appends
    layers = binding.LayerSet([{"cache": caches[0], "q": w.q.cuda(), "out": outs[0]},
                               {"cache": caches[2], "q": w.q.cuda(), "out": outs[1], "k_new": k_new, "v_new": v_new, "slot_mapping": slots}])
    layers.kv_stride = 2 * d
    binding.decode_layers(layers, table, lens_t, 6, w.sm_scale, plan, ws)
    assert torch.equal(outs[0], want) and torch.equal(outs[1], want) and torch.equal(caches[2].data, caches[0].data)
