"""The calls that a serving program makes of this library, as cases to be timed and compared.

Every case goes through the public binding (``paper_2602_09323_b200.binding``) the way a serving loop does: the
cache, the workspace, the plan buffer and the output buffers are kept from call to call, and one pass is one
call (or the few calls) that such a loop makes with what it has in hand.  Values follow the recipe of the
package's own workloads (N(0, 1) in bf16, two channels per head times 20), physical blocks are placed at random,
and every cache is filled through ``kv_write`` itself.

Kinds of pass:
  write     kv_write of a call's tokens: a few appended tokens per sequence, or the K/V of whole prompts
  step      decode_step: one layer's new tokens written, then attention, nothing planned beforehand
  decode    paged_decode over a cache that is there
  planned   decode_plan once, then decode_step_planned for every layer (a model step whose layers come one by one)
  layers    decode_layers over all layers in one call
  host      decode_step_host from page-locked host buffers, with the result awaited
  chunked   paged_chunked with one query token per sequence and its exported chunk partials (long contexts)
  prefill   the prompt chunk's K/V written with kv_write, then paged_chunked over old and new tokens
"""
import math
import random

import torch

from paper_2602_09323_b200 import binding

BLOCK = binding.BLOCK_SIZE
FORMATS = {"e4m3": binding.KV_FP8_E4M3, "e5m2": binding.KV_FP8_E5M2, "bf16": binding.KV_BF16}


def _case(name, kind, batch, lo, hi, hq, hkv, dim, **more):
    """``lo`` .. ``hi``: context lengths after the call, spread over the sequences (drawn from ``mix``)."""
    c = {"name": name, "kind": kind, "batch": batch, "lo": lo, "hi": hi, "hq": hq, "hkv": hkv, "dim": dim,
         "format": "e4m3", "layers": 1, "new": 1, "mix": 1, "chunk": 0, "overlap": False}
    c.update(more)
    return c


def listed():
    return [
        # one more token for each of a few dozen running sequences, at odd places of their blocks: the smallest call
        _case("append_tokens", "write", 48, 100, 2000, 40, 8, 128, mix=3),
        # a single user's chat turn: nothing to fill the GPU with, all latency
        _case("one_sequence_step", "step", 1, 777, 777, 40, 8, 128),
        # a full batch at equal lengths, all layers of a pipeline stage in one call: the package's own headline shape
        _case("layers_32x2048", "layers", 32, 2048, 2048, 40, 8, 128, layers=8, overlap=True),
        # a serving step over requests of very different lengths, layer by layer with the model's other work between
        _case("mixed_lengths_step", "planned", 64, 128, 8192, 40, 8, 128, layers=4, mix=5),
        # the common eight heads to a group, medium lengths
        _case("group_of_eight", "layers", 24, 300, 4000, 64, 8, 128, layers=4, mix=7, overlap=True),
        # a small model (head_dim 64) with many short requests, the other FP8 format
        _case("short_dim64_e5m2", "decode", 120, 5, 900, 16, 4, 64, format="e5m2", mix=9),
        # four very long documents, chunk partials exported
        _case("long_context", "chunked", 4, 32768, 131072, 40, 8, 128, chunk=2048, mix=0),
        # the step of a program that keeps its tensors on the host
        _case("host_step", "host", 32, 1900, 2100, 40, 8, 128, mix=11),
        # prompts taken in by chunks of 512 behind 4096 cached tokens
        _case("prefill_chunk", "prefill", 8, 4608, 4608, 40, 8, 128, new=512, chunk=2048),
        # whole prompts of a small model, ragged, nothing cached yet
        _case("prompts_dim64", "prefill", 4, 900, 2900, 32, 8, 64, new=0, chunk=2048, mix=13),
        # the cache of a full batch written at once (a restart, or K/V that come from elsewhere)
        _case("bulk_fill", "write", 32, 2048, 2048, 40, 8, 128, new=0),
        # the cache left in bf16, one kv head per query head
        _case("bf16_heads", "decode", 32, 2048, 2048, 40, 40, 128, format="bf16"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: any kind, group sizes 1 to 8, both head dims, short and long, odd sizes throughout."""
    while True:
        kind = rng.choice(["write", "step", "decode", "planned", "layers", "layers", "host", "chunked", "prefill", "prefill"])
        dim = rng.choice([128, 128, 128, 64])
        hkv = rng.choice([1, 2, 4, 8, 8])
        hq = hkv * rng.choice([1, 2, 4, 5, 5, 7, 8])
        batch = _log(rng, 1, 128)
        hi = _log(rng, 20, 131072 if kind == "chunked" else 8192)
        lo = rng.choice([hi, max(1, hi // 2), max(1, hi // 30)])
        more = {"mix": rng.randrange(1, 1000), "new": 1}
        if kind in ("planned", "layers"):
            more.update(layers=rng.choice([1, 3, 4, 8]), overlap=rng.random() < 0.5)
        if kind == "chunked":
            more["chunk"] = rng.choice([512, 2048])
            batch = min(batch, 16)
        if kind == "prefill":
            more.update(chunk=2048, new=rng.choice([0, _log(rng, 8, 1024)]))
            batch = max(2, min(batch, 24))
        if kind == "write":
            more["new"] = rng.choice([0, 1, _log(rng, 2, 600)])
        if kind in ("decode", "step", "write") and rng.random() < 0.25:
            more["format"] = "bf16"
        elif rng.random() < 0.2 and not (kind == "prefill" and dim == 64):
            more["format"] = "e5m2"
        c = _case("", kind, batch, lo, hi, hq, hkv, dim, **more)
        del c["name"]
        w = work(c)
        flops = 9e10 if dim == 64 else 3.5e11          # no dearer than the listed prompts and chunks
        if w["bytes"] <= 1.3e9 and (kind != "prefill" or w["flops"] <= flops) and sum(_lens(c)) <= 400000:
            return c


# ---- sizes -------------------------------------------------------------------------------------------------------

def _lens(c):
    """The context lengths, new tokens included."""
    if c["kind"] == "chunked" and c["mix"] == 0:      # an even ladder from lo to hi
        n = max(1, c["batch"] - 1)
        return [c["lo"] + (c["hi"] - c["lo"]) * i // n for i in range(c["batch"])]
    rng = random.Random(c["mix"])
    return [rng.randint(c["lo"], c["hi"]) for _ in range(c["batch"])]


def _new(c):
    """Tokens of each sequence that the pass brings (new = 0: all of them)."""
    lens = _lens(c)
    if c["kind"] == "prefill" and c["new"] > 1:       # chunks of prompts are ragged too, except where lengths are equal
        rng = random.Random(c["mix"] + 1)
        return [min(L, c["new"] if c["lo"] == c["hi"] else rng.randint(max(2, c["new"] // 3), c["new"])) for L in lens]
    return [L if c["new"] == 0 else min(L, c["new"]) for L in lens]


def work(case):
    lens, new, hkv, hq, d, layers = _lens(case), _new(case), case["hkv"], case["hq"], case["dim"], case["layers"]
    fp8 = case["format"] != "bf16"
    blocks = sum(-(-L // BLOCK) for L in lens)
    written = sum(-(-L // BLOCK) - (L - n) // BLOCK for L, n in zip(lens, new))
    token = 2 * hkv * d * (1 if fp8 else 2)                        # K and V of one token in the cache
    scales = 8 * hkv if fp8 else 0                                 # of one block
    io = 2 * hq * d * 2                                            # one token's query and output
    write = sum(new) * (2 * hkv * d * 2 + 8 + token) + written * scales
    kind = case["kind"]
    if kind == "write":
        return {"bytes": write, "flops": 0}
    read = sum(lens) * token + blocks * (scales + 4) + case["batch"] * 4
    if kind in ("step", "host", "planned", "layers"):
        return {"bytes": layers * (write + read + case["batch"] * io), "flops": layers * 4 * d * hq * sum(lens)}
    if kind == "decode":
        return {"bytes": read + case["batch"] * io, "flops": 4 * d * hq * sum(lens)}
    if kind == "chunked":
        chunks = sum(-(-L // case["chunk"]) for L in lens)
        return {"bytes": read + case["batch"] * io + chunks * hq * (d + 2) * 4, "flops": 4 * d * hq * sum(lens)}
    seen = sum(n * (L - n) + n * (n + 1) // 2 for L, n in zip(lens, new))          # (query, visible key) pairs
    return {"bytes": write + read + sum(new) * io, "flops": 4 * d * hq * seen}


def tolerance(case):
    if case["kind"] == "write":
        return "exact"
    # Measured against float64 attention over the same cache, rounded to bf16 once: the FP8 paths differ from it by
    # 1.0e-3 on average and 1.7e-3 at most (probabilities of 11 bits, then bf16 ties that fall the other way), single
    # values by 0.0125; the bf16 cache's path by 3e-4 and 0.0052.  Four times that.
    return {"rel": 1.3e-3, "max": 0.03} if case["format"] == "bf16" else {"rel": 7e-3, "max": 0.05}


# ---- inputs ------------------------------------------------------------------------------------------------------

class _Inputs:
    """Seeded inputs of one case on the GPU: block placement, and values in the package's recipe."""

    def __init__(self, case, seed):
        self.c = case
        self.gen = torch.Generator(device="cuda").manual_seed(seed)
        self.lens, self.new = _lens(case), _new(case)
        need = [-(-L // BLOCK) for L in self.lens]
        self.width = max(need)
        self.num_blocks = sum(need) + max(1, sum(need) // 10)
        place = torch.randperm(self.num_blocks, generator=self.gen, device="cuda").to(torch.int32)
        at, rows = 0, []
        for n in need:
            rows.append(torch.nn.functional.pad(place[at:at + n], (0, self.width - n), value=-1))
            at += n
        self.table = torch.stack(rows).contiguous()
        self.lens_t = torch.tensor(self.lens, dtype=torch.int32, device="cuda")
        self.scale = 1.0 / math.sqrt(case["dim"])

    def values(self, rows, heads):
        x = torch.randn(rows, heads, self.c["dim"], generator=self.gen, device="cuda", dtype=torch.bfloat16)
        loud = torch.rand(heads, self.c["dim"], generator=self.gen, device="cuda").topk(2, dim=1).indices
        return x * torch.ones(heads, self.c["dim"], device="cuda", dtype=torch.bfloat16).scatter_(1, loud, 20.0)

    def slots(self, spans):
        """Slots of positions start .. stop - 1 of every sequence, one sequence after the other."""
        got = []
        for b, (start, stop) in enumerate(spans):
            pos = torch.arange(start, stop, device="cuda")
            got.append(self.table[b, pos // BLOCK].long() * BLOCK + pos % BLOCK)
        return torch.cat(got)

    def cache(self, held):
        """A cache that holds the first ``held[b]`` tokens of every sequence."""
        cache = binding.Cache(self.num_blocks, self.c["hkv"], self.c["dim"], FORMATS[self.c["format"]])
        if sum(held):
            n = sum(held)
            binding.kv_write(cache, self.values(n, self.c["hkv"]), self.values(n, self.c["hkv"]), self.slots([(0, h) for h in held]))
        return cache

    def workspace(self, chunk=0):
        c = self.c
        return binding.new_workspace(c["batch"], c["hq"], c["hkv"], c["dim"], self.width, chunk, sum(self.new))


def prepare(case, seed):
    i, c = _Inputs(case, seed), case
    kind, hq, hkv, d, batch = c["kind"], c["hq"], c["hkv"], c["dim"], c["batch"]
    s = {"kind": kind, "case": c, "table": i.table, "lens": i.lens_t, "scale": i.scale, "width": i.width}
    old = [L - n for L, n in zip(i.lens, i.new)]
    fresh = lambda: (i.values(sum(i.new), hkv), i.values(sum(i.new), hkv))
    slots = i.slots(list(zip(old, i.lens)))
    if kind in ("planned", "layers"):
        s["out"] = torch.empty(c["layers"], batch, hq, d, dtype=torch.bfloat16, device="cuda")
        s["layers"] = []
        for l in range(c["layers"]):
            cache = i.cache(old)
            k, v = fresh()
            s["layers"].append({"cache": cache, "k_new": k, "v_new": v, "slot_mapping": slots, "q": i.values(batch, hq), "out": s["out"][l]})
        s["set"] = binding.LayerSet(s["layers"])
        s["ws"] = i.workspace()
        s["plan"] = torch.empty(binding.plan_bytes(batch, hkv, i.width), dtype=torch.uint8, device="cuda")
        return s
    s["cache"] = i.cache(i.lens if kind in ("decode", "chunked") else old)
    if kind not in ("decode", "chunked"):
        s["k"], s["v"] = fresh()
        s["slots"] = slots
    if kind == "write":
        return s
    s["ws"] = i.workspace(c["chunk"])
    rows = sum(i.new) if kind == "prefill" else batch
    q = s["q"] = i.values(rows, hq)
    s["out"] = torch.empty_like(q)
    if kind in ("chunked", "prefill"):
        n = i.new if kind == "prefill" else [1] * batch
        s["cu"] = torch.tensor([0] + n, dtype=torch.int32, device="cuda").cumsum(0).to(torch.int32)
    if kind == "chunked":      # where the calls leave the (o, m, l) of every chunk that exists
        o, m, l = binding.chunk_partials(s["ws"], batch, hq, d, i.width, c["chunk"])
        chunks = [-(-L // c["chunk"]) for L in i.lens]
        s["partials"] = [x[b, :, :n] for b, n in enumerate(chunks) for x in (o, m, l)]
    if kind == "host":
        lay = binding.step_staging_layout(batch, hq, hkv, d, i.width)
        packed = torch.zeros(lay.in_bytes, dtype=torch.uint8)
        for at, t in ((lay.q, q), (lay.k_new, s["k"]), (lay.v_new, s["v"]), (lay.slot_mapping, slots), (lay.block_table, i.table),
                      (lay.context_lens, i.lens_t)):
            raw = t.cpu().contiguous().view(torch.uint8).reshape(-1)
            packed[at:at + raw.numel()] = raw
        s["in"], s["out"] = packed.pin_memory(), torch.empty(batch, hq, d, dtype=torch.bfloat16).pin_memory()
        s["staging"] = torch.empty(lay.total_bytes, dtype=torch.uint8, device="cuda")
        s["plan"] = torch.empty(binding.plan_bytes(batch, hkv, i.width), dtype=torch.uint8, device="cuda")
    return s


# ---- one pass ----------------------------------------------------------------------------------------------------

def run(state):
    s, c = state, state["case"]
    kind = s["kind"]
    flags = binding.FLAG_OVERLAP_PREVIOUS if c["overlap"] else 0
    if kind == "layers":
        binding.decode_layers(s["set"], s["table"], s["lens"], c["hq"], s["scale"], s["plan"], s["ws"], flags)
        return [s["out"]] + [L["cache"].data for L in s["layers"]]
    if kind == "planned":
        binding.decode_plan(s["table"], s["lens"], c["hkv"], s["layers"][0]["cache"].num_blocks, plan=s["plan"])
        for n, L in enumerate(s["layers"]):
            binding.decode_step_planned(L["cache"], s["plan"], L["q"], s["width"], s["scale"], s["ws"], L["k_new"], L["v_new"],
                                        L["slot_mapping"], flags=flags if n else 0, out=L["out"])
        return [s["out"]] + [L["cache"].data for L in s["layers"]]
    if kind == "write":
        binding.kv_write(s["cache"], s["k"], s["v"], s["slots"])
        return s["cache"].data
    if kind == "step":
        out = binding.decode_step(s["cache"], s["k"], s["v"], s["slots"], s["q"], s["table"], s["lens"], s["scale"], s["ws"], out=s["out"])
        return [out, s["cache"].data]
    if kind == "decode":
        return binding.paged_decode(s["cache"], s["q"], s["table"], s["lens"], s["scale"], s["ws"], out=s["out"])
    if kind == "host":
        binding.decode_step_host(s["cache"], s["in"], s["out"], s["width"], c["hq"], s["scale"], s["staging"], s["plan"], s["ws"])
        torch.cuda.current_stream().synchronize()        # the program reads its result on the host
        return [s["out"], s["cache"].data]
    if kind == "prefill":
        binding.kv_write(s["cache"], s["k"], s["v"], s["slots"])
        out = binding.paged_chunked(s["cache"], s["q"], s["cu"], s["table"], s["lens"], c["chunk"], True, s["scale"], s["ws"], out=s["out"])
        return [out, s["cache"].data]
    out = binding.paged_chunked(s["cache"], s["q"], s["cu"], s["table"], s["lens"], c["chunk"], True, s["scale"], s["ws"], out=s["out"])
    return [out] + s["partials"]
