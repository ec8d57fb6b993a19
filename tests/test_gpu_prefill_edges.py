"""GPU parity of the prefill kernel where its tiling can go wrong: query runs around the edges of a tile and of a pair of
tiles, contexts around the edges of a tile of keys, one pair of which a tile sees fewer keys, every group size's tile."""
import pytest
import torch

from oracle import attention
from paper_2602_09323_b200 import binding, workloads
from tests import helpers

pytestmark = pytest.mark.gpu


def _check(lens, q_lens, hq, hkv, d, causal=True, seed=0, mutate=None):
    w = workloads.make_workload("prefill_edges", lens, hq, hkv, d, seed=seed, q_lens=q_lens)
    if mutate:
        mutate(w)
    cache = helpers.gpu_fill(w)
    ws = binding.new_workspace(w.batch, hq, hkv, d, w.block_table.shape[1], 2048, sum(q_lens))
    call = lambda: binding.paged_chunked(cache, w.q.cuda(), w.cu_q_lens.cuda(), w.block_table.cuda(), w.context_lens_tensor.cuda(), 2048, causal, w.sm_scale, ws)
    out = call()
    torch.cuda.synchronize()
    assert binding.workspace_status(ws) == 0
    ref = attention.paged_attention(w.q.float().numpy(), helpers.oracle_fp8_cache(w), w.block_table.numpy(), w.context_lens,
                                    cu_q_lens=w.cu_q_lens.numpy(), causal=causal)
    helpers.check_attention(out, ref, what=f"prefill {lens} {q_lens}")      # the repository's bound: bf16 output, 11-bit probabilities
    assert torch.equal(out, call())


@pytest.mark.parametrize("hq,hkv,d", [(1, 1, 128), (5, 1, 128), (8, 1, 64), (3, 1, 64), (2, 1, 128)])
def test_query_runs_around_tile_edges(hq, hkv, d):
    tq = 128 // (hq // hkv)
    q_lens = [1, tq - 1, tq, tq + 1, 2 * tq - 1, 2 * tq, 2 * tq + 1]
    _check([n + 130 for n in q_lens], q_lens, hq, hkv, d, seed=hq)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("causal", [True, False])
def test_contexts_around_key_tile_edges(d, causal):
    lens = [16, 127, 128, 129, 143, 144, 145, 255, 256, 257, 513, 641]
    _check(lens, [min(n, 40) for n in lens], 4, 2, d, causal=causal, seed=d)


@pytest.mark.parametrize("d", [64, 128])
def test_a_first_tile_that_sees_fewer_key_tiles_than_the_second(d):
    _check([256, 300, 520], [256, 200, 250], 1, 1, d, seed=7)                # 128 queries a tile: one key tile apart


@pytest.mark.parametrize("d", [64, 128])
def test_references_that_have_to_move(d):
    """Logits that grow along the context by far more than the margin of a lazy maximum, V scales by more than theirs."""
    def mutate(w):
        n = w.k.shape[0]
        grow = torch.linspace(0.01, 3.0, n)[:, None, None]
        w.k[:] = (w.k.float() * grow).to(torch.bfloat16)
        w.v[:] = (w.v.float() * (torch.arange(n)[:, None, None] // 200 * 2.0 + 0.01) * 0.02).to(torch.bfloat16)
    _check([900, 700], [100, 30], 6, 2, d, seed=9, mutate=mutate)


@pytest.mark.parametrize("batch", [3, 33, 128, 129])
def test_more_tiles_than_the_device_holds_ragged(batch):
    """Every (sequence, kv head, pair of tiles) is found once in the order of lengths, with sequences whose runs are empty or
    longer than their context's start, on both sides of the number of sequences that are ordered."""
    g = torch.Generator().manual_seed(batch)
    lens = [int(n) for n in torch.randint(1, 260, (batch,), generator=g)]
    q_lens = [0 if i % 7 == 3 else max(1, n - (37 * i) % 90) for i, n in enumerate(lens)]
    if batch == 3:
        lens, q_lens = [700, 40, 1500], [690, 40, 900]
    _check(lens, q_lens, 32, 4, 64, seed=batch)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("sm_scale", [-0.0625, -1.0, 0.0])
def test_a_logit_scale_that_is_not_positive(d, sm_scale):
    """As in decode: the logits are scaled by what the caller gives, its sign included, which is the same as -q and the other
    sign.  (A scale of 1 is not held against the oracle: at head_dim 128 a logit's error is up to sm_scale 2^-17 max|q| sum|k|,
    here 2^-17 * 60 * 130 = 0.06 of a probability; of 1/16, 0.004.)"""
    w = workloads.make_workload("negative", [300, 140, 17], 6, 2, d, seed=d, q_lens=[100, 33, 17])
    cache, ws = helpers.gpu_fill(w), binding.new_workspace(w.batch, 6, 2, d, w.block_table.shape[1], 2048, 150)
    for causal in (True, False):
        call = lambda q, s: binding.paged_chunked(cache, q, w.cu_q_lens.cuda(), w.block_table.cuda(), w.context_lens_tensor.cuda(), 2048, causal, s, ws)
        out = call(w.q.cuda(), sm_scale)
        torch.cuda.synchronize()
        assert binding.workspace_status(ws) == 0
        assert torch.equal(out, call(-w.q.cuda(), -sm_scale))
        if sm_scale == -1.0:
            continue
        ref = attention.paged_attention(w.q.float().numpy(), helpers.oracle_fp8_cache(w), w.block_table.numpy(), w.context_lens,
                                        cu_q_lens=w.cu_q_lens.numpy(), causal=causal, sm_scale=sm_scale)
        helpers.check_attention(out, ref, what=f"prefill, logits times {sm_scale}")


@pytest.mark.parametrize("hq,hkv,d", [(16, 16, 128), (60, 12, 128), (96, 12, 64)])
def test_query_runs_around_the_edges_of_pairs_of_tiles(hq, hkv, d):
    """As test_query_runs_around_tile_edges, with so many kv heads that a CTA has two tiles."""
    test_query_runs_around_tile_edges(hq, hkv, d)


@pytest.mark.parametrize("d", [64, 128])
def test_a_first_tile_of_a_pair_that_sees_fewer_key_tiles_than_the_second(d):
    _check([256, 300, 520], [256, 200, 250], 20, 20, d, seed=7)


@pytest.mark.parametrize("more", [0, 1])
@pytest.mark.parametrize("d", [64, 128])
def test_on_both_sides_of_as_many_tiles_as_multiprocessors(d, more):
    """16 queries a tile; the launch reckons with one tile more than the sequence fills."""
    n = 16 * (torch.cuda.get_device_properties(0).multi_processor_count - 1 + more)
    _check([n + 5], [n], 8, 1, d, seed=more)


@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("hkv,d", [(20, 64), (20, 128), (2, 64), (2, 128)])
def test_runs_of_one_to_five_tiles_with_and_without_turns(hkv, d, causal):
    """From the start of their context and behind others: with twenty kv heads a CTA has two tiles, which take turns at the
    exponentials, as long and unequally long as they come; with two it has one, by another kernel.  (Without loud channels: at
    head_dim 128 a logit's error is up to sm_scale 2^-17 max|q| sum|k|, with them 2^-17 * 80 * 160 / 11.3 = 0.009 of a
    probability, and of values of 80 among 4.8 million one is off by 0.05; without 2^-17 * 5.5 * 130 / 11.3 = 0.0005.)"""
    def mutate(w):
        for x in (w.q, w.k, w.v):
            x.clamp_(-5.5, 5.5)
    _check([64, 65, 128, 300, 300, 500], [64, 65, 128, 129, 300, 257], 2 * hkv, hkv, d, causal=causal, seed=d + hkv, mutate=mutate)
