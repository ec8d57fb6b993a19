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
