"""Where the time of one launch goes: ``python -m paper_2602_09323_b200.trace [--workload ...]``.

Builds ``libcoopt_trace.so`` (the library's sources with ``-DCOOPT_TRACE``), runs the fused decode step of a
workload a few times and prints, for the last launch, when the decode kernel's CTAs reached their
milestones: per milestone the median, the earliest and the latest CTA, in microseconds from that CTA's own
first instruction, and the span of the whole launch on the global timer.  The stamps cost a few stores, so this is a
breakdown, not a benchmark.
"""
from __future__ import annotations

import argparse
import ctypes

import numpy as np
import torch

from . import binding, build, workloads

SLOTS = 32
MAX_CTAS = 1024
ENTRY, ENTRY_NS, STREAMED, EXIT, EXIT_NS, SM_ID, PREV_EXIT_NS, BLOCKS, WARP_END = 0, 1, 7, 8, 9, 10, 11, 12, 16
MILESTONES = {2: "line_summed", 3: "first_copies", 4: "previous_done", 5: "query_ready", 6: "first_landed", STREAMED: "streamed", EXIT: "exit"}
SHAPES = {"one_sequence": ([777], 40, 8, 128), "short": ([3, 28, 17, 9, 22, 28, 1, 14], 56, 8, 128), "group_of_eight": (None, 64, 8, 128)}


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--workload", default="llama13b_decode",
                    choices=["llama13b_decode", "mixed_serving", "long_context"] + sorted(SHAPES))
    ap.add_argument("--no-append", action="store_true", help="attention only (no new token written in the launch)")
    ap.add_argument("--overlap", action="store_true", help="every launch may start while the one before it drains")
    ap.add_argument("--launches", type=int, default=12)
    ap.add_argument("--per-cta", action="store_true", help="also list every CTA: SM, blocks of warp 0, life time")
    ap.add_argument("--sm-mhz", type=float, default=1965.0, help="SM clock used to turn cycles into microseconds")
    args = ap.parse_args()
    binding.use_library(build.build(trace=True))
    lib = binding.load_library()
    lib.coopt_trace_set_buffer.restype, lib.coopt_trace_set_buffer.argtypes = ctypes.c_int, [ctypes.c_void_p, ctypes.c_size_t]
    torch.cuda.set_device(0)
    chunk = 0
    if args.workload == "llama13b_decode":
        w = workloads.config_llama13b_decode()
    elif args.workload == "mixed_serving":
        w = workloads.config_mixed_serving()
    elif args.workload == "long_context":
        w, chunk = workloads.config_long_context(), 2048
    else:
        lengths, hq, hkv, d = SHAPES[args.workload]
        w = workloads.make_workload(args.workload, lengths or workloads.uniform_lengths(24, 300, 4000, 7), hq, hkv, d)
    B, Hq, Hkv, D = w.batch, w.num_q_heads, w.num_kv_heads, w.head_dim
    k, v, slots = w.k.cuda(), w.v.cuda(), w.slot_mapping.cuda()
    last = torch.tensor([w.kv_offsets[b] + L - 1 for b, L in enumerate(w.context_lens)])
    hist = torch.ones(k.shape[0], dtype=torch.bool)
    hist[last] = False
    hist_idx, new_idx = hist.nonzero().squeeze(1).cuda(), last.cuda()
    k_new, v_new, s_new = k[new_idx].contiguous(), v[new_idx].contiguous(), slots[new_idx].contiguous()
    caches = []
    for _ in range(2):                      # two caches visited in turn: more than L2 between two visits of one
        c = binding.Cache(w.num_blocks, Hkv, D)
        binding.kv_write(c, k[hist_idx], v[hist_idx], slots[hist_idx])
        caches.append(c)
    table, lens, q = w.block_table.clamp(min=0).cuda(), w.context_lens_tensor.cuda(), w.q.cuda()
    plan = binding.decode_plan(table, lens, Hkv, w.num_blocks, chunk)
    ws = binding.new_workspace(B, Hq, Hkv, D, table.shape[1], chunk, B)
    buf = torch.zeros(MAX_CTAS * SLOTS, dtype=torch.int64, device="cuda")
    assert lib.coopt_trace_set_buffer(ctypes.c_void_p(buf.data_ptr()), buf.numel() * 8) == 0
    out = torch.empty_like(q)
    new = (None, None, None) if args.no_append else (k_new, v_new, s_new)
    torch.cuda.synchronize()
    for i in range(args.launches):          # (every launch follows its predecessor directly and finds its exit times)
        binding.decode_step_planned(caches[i % 2], plan, q, table.shape[1], w.sm_scale, ws, *new, chunk_size=chunk, out=out,
                                    flags=binding.FLAG_OVERLAP_PREVIOUS if args.overlap and i else 0)
    torch.cuda.synchronize()
    assert binding.workspace_status(ws) == 0
    t = buf.cpu().numpy().reshape(MAX_CTAS, SLOTS)
    t = t[t[:, ENTRY] != 0]
    us = 1.0 / args.sm_mhz
    if args.per_cta:
        print("CTA   SM  blocks of warp 0  first landed  streamed  exit (us)")
        for i, x in enumerate(t):
            print(f"{i:4d} {int(x[SM_ID]) - 1:4d} {int(x[BLOCKS]):4d}  {(x[6] - x[0]) * us:8.2f} {(x[STREAMED] - x[0]) * us:8.2f} {(x[EXIT] - x[0]) * us:8.2f}")
    print(f"workload {args.workload}{' (no append)' if args.no_append else ''}{' (overlapped)' if args.overlap else ''}: {t.shape[0]} CTAs, "
          f"blocks of warp 0 median {np.median(t[:, BLOCKS]):.0f} max {t[:, BLOCKS].max()}")
    print(f"launch span on the global timer: {(t[:, EXIT_NS].max() - t[:, ENTRY_NS].min()) / 1e3:.1f} us (first entry to last exit); entries spread "
          f"over {(t[:, ENTRY_NS].max() - t[:, ENTRY_NS].min()) / 1e3:.1f} us, exits over {(t[:, EXIT_NS].max() - t[:, EXIT_NS].min()) / 1e3:.1f} us")
    if t[:, PREV_EXIT_NS].min() > 0:
        print(f"last exit of the launch before to first entry of this one: {(t[:, ENTRY_NS].min() - t[:, PREV_EXIT_NS].max()) / 1e3:.2f} us; "
              f"to last exit of this one: {(t[:, EXIT_NS].max() - t[:, PREV_EXIT_NS].max()) / 1e3:.2f} us")
    print(f"{'milestone':<16}{'median':>9}{'earliest':>10}{'latest':>9}   (us after the CTA's first instruction, {args.sm_mhz:.0f} MHz)")
    ends = t[:, WARP_END:WARP_END + 16]
    cols = [(name, t[:, i]) for i, name in MILESTONES.items()]
    cols[-2:-2] = [("first_warp_done", np.where(ends > 0, ends, np.iinfo(np.int64).max).min(axis=1)), ("last_warp_done", ends.max(axis=1))]
    for name, col in cols:
        ok = col != 0
        if ok.any():
            rel = (col[ok] - t[ok, ENTRY]) * us
            print(f"{name:<16}{np.median(rel):9.2f}{rel.min():10.2f}{rel.max():9.2f}   ({int(ok.sum())} CTAs)")


if __name__ == "__main__":
    main()
