"""Bulk writes (more than 512 tokens) against the oracle, bit for bit, where the split into blocks that are written whole and
others can go wrong: sequences that begin and end anywhere, whole blocks across the edges of a 32-token span, skipped
tokens, tokens out of order inside a block, strides and addresses that only suit element loads, extreme scales, zeros of
both signs, every head dim and format."""
import numpy as np
import pytest
import torch

from oracle import e5m2, kv_cache
from paper_2602_09323_b200 import binding, workloads
from tests import helpers

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,fmt,hkv", [(128, "e4m3", 5), (64, "e4m3", 2), (128, "e5m2", 1), (64, "e5m2", 3)])
@pytest.mark.parametrize("how", ["ragged", "skips", "shuffled in blocks", "odd stride", "extreme"])
def test_bulk_write_bit_exact(d, fmt, hkv, how):
    lens = [1, 16, 17, 31, 100, 333, 15, 64, 9, 240]
    w = workloads.make_workload("bulk", lens, hkv, hkv, d, seed=d + hkv)
    k, v, slots = w.k.clone(), w.v.clone(), w.slot_mapping.clone()
    gen = torch.Generator().manual_seed(3)
    if how == "skips":
        slots[torch.randperm(len(slots), generator=gen)[:60]] = -1
    if how == "shuffled in blocks":
        order = torch.arange(len(slots))
        for i in range(0, 300, 16):                      # tokens of a block stay consecutive, their order changes
            at = w.kv_offsets[5] + i
            n = min(16, w.kv_offsets[5] + 333 - at)
            order[at:at + n] = at + torch.randperm(n, generator=gen)
        k, v, slots = k[order], v[order], slots[order]
    if how == "extreme":
        k[:, :, ::3] = -0.0
        v[40:60] = 0.0
        v[60:64] = -0.0
        k[100:200] *= 2.0 ** -50
        v[200:300] *= 2.0 ** 60
        k[300:340] = torch.tensor(2.0 ** -133).to(torch.bfloat16)
    cache = binding.Cache(w.num_blocks, hkv, d, binding.KV_FP8_E5M2 if fmt == "e5m2" else binding.KV_FP8_E4M3)
    if how == "odd stride":                              # rows an odd number of elements apart: no aligned row
        store = torch.zeros(2, len(slots) * (hkv * d + 1) + 1, dtype=torch.bfloat16, device="cuda")
        kd, vd = (store[i][1:].as_strided(k.shape, (hkv * d + 1, d, 1)) for i in range(2))
        kd.copy_(k), vd.copy_(v)
    else:
        kd, vd = k.cuda(), v.cuda()
    binding.kv_write(cache, kd, vd, slots.cuda())
    codes, scales = kv_cache.new_cache(w.num_blocks, hkv, d)
    kw = {"fmt": e5m2} if fmt == "e5m2" else {}
    kv_cache.kv_write(codes, scales, k.float().numpy(), v.float().numpy(), slots.numpy(), **kw)
    helpers.check_cache_bit_exact(cache, codes, scales, what=how)


@pytest.mark.parametrize("d,hkv,sequences,run", [(128, 1, 270, 2), (128, 1, 300, 13), (64, 5, 200, 7), (64, 5, 400, 13), (128, 5, 400, 11), (128, 4, 800, 20), (64, 1, 1500, 13)])
def test_short_runs_of_many_sequences_in_two_calls(d, hkv, sequences, run):
    """Spans that 16, 8, 4, 2 CTAs share and that one CTA has alone; the second call finds codes in the blocks."""
    w = workloads.make_workload("runs", [2 * run] * sequences, hkv, hkv, d, seed=run)
    first = np.concatenate([np.arange(o, o + run) for o in w.kv_offsets])
    helpers.check_cache_bit_exact(helpers.gpu_fill(w, calls=[first, first + run]), *helpers.oracle_fp8_cache(w, calls=[first, first + run]))
