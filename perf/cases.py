"""Speed cases of the eviction hot path: prompt compression (he_prefill_compress) and the decode loop (he_decode_step, with
or without the attention over the compressed cache that follows it), called as a user's program calls them.

A case is a flat dict:
  op          "prefill": one HashEvictCache.prefill_compress over a batch of prompts
              "decode": `tokens` tokens, each taken through `layers` layers (one cache and one W per layer), per layer a
              decode_step and, with `attend`, the attention over the cache that the step left
  batch, kv_heads, group, dim, bits, dtype    shape of a layer
  budget_lo, budget_hi    cache budget per sequence, uniform in that range (equal: the same for all)
  prompt      prompt length per sequence as a multiple of its budget, in thousandths (2000: twice the budget, the 50 % setting)
  keys        "iid" | "drift" (4 outlier channels x 10 per head, slow mean drift) | "cluster" (16 Gaussian clusters, outliers)
  sink, recent    protected windows
  layers, tokens, attend, graph, early    decode only: `graph` replays a captured CUDA graph of the calls, as a serving loop
              does; otherwise every call is enqueued from Python. `early`: inputs staged ahead (HE_FLAG_EARLY_INPUTS).
"""
import math

import torch

from paper_2412_16187_b200 import HashEvictCache

_DT = {"bf16": torch.bfloat16, "f32": torch.float32}


def _prefill(name, batch, kv_heads, group, dim, bits, dtype, budget_lo, budget_hi, prompt, keys, sink=0, recent=0):
    return {"name": name, "op": "prefill", "batch": batch, "kv_heads": kv_heads, "group": group, "dim": dim, "bits": bits, "dtype": dtype,
            "budget_lo": budget_lo, "budget_hi": budget_hi, "prompt": prompt, "keys": keys, "sink": sink, "recent": recent}


def _decode(name, batch, kv_heads, group, dim, bits, dtype, budget_lo, budget_hi, prompt, keys, layers, tokens, attend, graph, early,
            sink=0, recent=0):
    c = _prefill(name, batch, kv_heads, group, dim, bits, dtype, budget_lo, budget_hi, prompt, keys, sink, recent)
    c.update(op="decode", layers=layers, tokens=tokens, attend=attend, graph=graph, early=early)
    return c


def listed():
    return [
        # --- decode
        # the tiny configuration, one call enqueued from Python: nothing but launch and host latency
        _decode("decode tiny fp32", 1, 4, 1, 64, 8, "f32", 64, 64, 2000, "iid", 1, 1, False, False, False),
        # one multi-head layer stepped from a Python loop: evict, then attend over 2048 slots
        _decode("decode mha layer + attend", 1, 32, 1, 128, 32, "bf16", 2048, 2048, 2000, "drift", 1, 1, True, False, False),
        # grouped-query batch of 16 with the protected windows that the paper's runs use, 8 layers, captured
        _decode("decode gqa x16, protected", 16, 8, 4, 128, 16, "bf16", 1024, 1024, 8000, "drift", 8, 4, False, True, False, 4, 10),
        # long context at batch 1: 9830 slots per head, evict and attend layer by layer, captured
        _decode("decode long + attend", 1, 8, 4, 128, 32, "bf16", 9830, 9830, 1333, "drift", 8, 4, True, True, False),
        # the throughput batch: 64 sequences with ragged budgets, 64-bit codes, inputs staged ahead, captured
        _decode("decode ragged x64, early", 64, 8, 4, 128, 64, "bf16", 512, 4096, 2000, "cluster", 8, 4, False, True, True),
        # the largest step: 256 sequences in one call, enqueued from Python
        _decode("decode ragged x256", 256, 8, 4, 128, 64, "bf16", 512, 4096, 1100, "cluster", 1, 1, False, False, False),
        # --- prompt compression
        _prefill("prefill tiny fp32", 1, 4, 1, 64, 8, "f32", 64, 64, 2000, "iid"),
        # one multi-head layer: a 4096-token prompt, half of it kept
        _prefill("prefill mha layer", 1, 32, 1, 128, 32, "bf16", 2048, 2048, 2000, "drift"),
        # grouped-query batch of 16, 8192-token prompts kept to an eighth, protected windows
        _prefill("prefill gqa x16, protected", 16, 8, 4, 128, 16, "bf16", 1024, 1024, 8000, "drift", 4, 10),
        # one layer of a long-context prompt (32768 tokens, 30 % kept): 8 units have the whole GPU
        _prefill("prefill long layer", 1, 8, 4, 128, 32, "bf16", 9830, 9830, 3334, "drift"),
        # the throughput batch: 64 prompts of 1024..8192 tokens, half of each kept
        _prefill("prefill ragged x64", 64, 8, 4, 128, 64, "bf16", 512, 4096, 2000, "cluster"),
        # the largest: the long-context prompt with its 32 layers folded into the batch
        _prefill("prefill long x32", 32, 8, 4, 128, 32, "bf16", 9830, 9830, 3334, "drift"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Shapes of a transformer layer (4 to 32 KV heads, groups of 1 to 8, head size 64 or 128), code lengths of the paper's
    sweep, budgets from 64 slots to the longest configuration's 9830, prompts 1.1 to 10 times the budget (10-90 % kept)."""
    while True:
        fp32 = rng.random() < 0.12
        keys = rng.choice(("iid", "drift", "drift", "cluster", "cluster"))
        hi = _log(rng, 64, 9830 if not fp32 else 2048)
        lo = rng.randint(max(48, hi // 8), hi) if rng.random() < 0.5 else hi
        prompt = _log(rng, 1111, 10000)
        sink, recent = rng.choice(((0, 0), (0, 0), (4, 10)))
        shape = (_log(rng, 1, 64), rng.choice((4, 8, 8, 32)), rng.choice((1, 2, 4, 4, 4, 8)), rng.choice((64, 128, 128, 128)),
                 rng.choice((8, 16, 24, 32, 32, 64, 64)), "f32" if fp32 else "bf16", lo, hi, prompt, keys)
        units, n = shape[0] * shape[1], hi * prompt // 1000
        if n > 32768:
            continue
        if rng.random() < 0.55:
            c = _prefill("", *shape, sink, recent)
            if units * n > 2_000_000 or units * n * (lo + hi) > 8_000_000_000:
                continue
        else:
            graph = rng.random() < 0.6
            c = _decode("", *shape, _log(rng, 1, 8) if graph else 1, rng.randint(1, 4) if graph else 1, rng.random() < 0.4, graph,
                        rng.random() < 0.5, sink, recent)
            # the prompt only fills the caches here: short, so that preparing takes little
            c["prompt"] = 1111 + prompt // 20
            if units * hi * c["layers"] * shape[3] > 4_000_000_000 or units * hi * c["prompt"] > 2_000_000_000:
                continue
        del c["name"]
        return c


def _lengths(case):
    """Budgets and prompt lengths of the sequences. Part of the case: two seeds of it differ in values only."""
    g = torch.Generator().manual_seed(case["budget_lo"] * 1_000_003 + case["budget_hi"])
    budgets = torch.randint(case["budget_lo"], case["budget_hi"] + 1, (case["batch"],), generator=g, dtype=torch.int64)
    return budgets, torch.clamp(budgets * case["prompt"] // 1000, max=32768)


class _Maker:
    """Post-RoPE-like K / Q / V: channel outliers, drift and clusters per head, as the synthetic workloads have them."""

    def __init__(self, case, seed):
        self.case, self.g = case, torch.Generator(device="cuda").manual_seed(seed)
        b, h, d = case["batch"], case["kv_heads"], case["dim"]
        self.scale = torch.ones((b, h, 1, d), device="cuda")
        if case["keys"] != "iid":
            at = torch.rand((b, h, 1, d), generator=self.g, device="cuda").topk(4, dim=3).indices
            self.scale.scatter_(3, at, 10.0)
        self.drift = torch.randn((b, h, 1, d), generator=self.g, device="cuda")
        self.centres = 2.0 * torch.randn((b, h, 16, d), generator=self.g, device="cuda") if case["keys"] == "cluster" else None

    def normal(self, *shape, dtype=None):
        return torch.randn(shape, generator=self.g, device="cuda", dtype=dtype or _DT[self.case["dtype"]])

    def keys(self, tokens, of):
        """[batch, kv_heads, tokens, dim], a sequence at a time to keep the temporaries small."""
        c = self.case
        out = torch.empty((c["batch"], c["kv_heads"], tokens, c["dim"]), device="cuda", dtype=_DT[c["dtype"]])
        for s in range(c["batch"]):
            z = self.normal(c["kv_heads"], tokens, c["dim"], dtype=torch.float32)
            if c["keys"] == "cluster":
                at = torch.randint(0, 16, (c["kv_heads"], tokens, 1), generator=self.g, device="cuda").expand(-1, -1, c["dim"])
                z.mul_(0.5).add_(torch.gather(self.centres[s], 1, at))
            z.mul_(self.scale[s])
            if c["keys"] == "drift":
                z.add_(self.drift[s] * (torch.arange(tokens, device="cuda").view(1, -1, 1) / of))
            out[s] = z
        return out


def prepare(case, seed):
    m = _Maker(case, seed)
    b, h, g, d, n_bits, dt = case["batch"], case["kv_heads"], case["group"], case["dim"], case["bits"], _DT[case["dtype"]]
    budgets, lens = _lengths(case)
    n = int(lens.max())
    decode = case["op"] == "decode"
    caches = [HashEvictCache(b, h, g, d, n_bits, budgets, m.normal(d, n_bits, dtype=torch.float32), dtype=dt, n_sink=case["sink"],
                             n_recent=case["recent"], early_inputs=bool(decode and case["early"]))
              for _ in range(case["layers"] if decode else 1)]
    k = m.keys(n, n + 64)
    v, q = m.normal(b, h, n, d), m.normal(b, h * g, n, d)
    state = {"case": case, "caches": caches, "prompt_len": lens.to(device="cuda", dtype=torch.int32), "n": n}
    if not decode:
        caches[0].workspace(n)
        state.update(q=q, k=k, v=v)
        return state
    ws = caches[0].workspace(n)
    for c in caches:
        c.prefill_compress(q, k, v, state["prompt_len"], n, workspace=ws)
    layers, tokens = len(caches), case["tokens"] if case["graph"] else 8
    dk = m.keys(layers * tokens, layers * tokens).permute(2, 0, 1, 3).contiguous().view(tokens, layers, b, h, d)
    state.update(tokens=tokens, at=0, dk=dk, dv=m.normal(tokens, layers, b, h, d), dq=m.normal(tokens, layers, b, h * g, d),
                 victim=torch.empty((case["tokens"], layers, b, h), dtype=torch.int32, device="cuda"),
                 evicted=torch.empty((case["tokens"], layers, b, h), dtype=torch.int32, device="cuda"),
                 out=torch.empty((case["tokens"], layers, b, h * g, d), device="cuda") if case["attend"] else None)
    torch.cuda.synchronize()
    if case["graph"]:
        state["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(state["graph"]):
            for t in range(tokens):
                _token(state, t, t)
    return state


def _token(state, t, to):
    """Token t of the staged inputs through every layer."""
    for i, c in enumerate(state["caches"]):
        q = state["dq"][t, i]
        c.decode_step(q, state["dk"][t, i], state["dv"][t, i], victim_out=state["victim"][to, i], evicted_pos_out=state["evicted"][to, i])
        if state["out"] is not None:
            c.attend(q, out=state["out"][to, i])


def run(state):
    if state["case"]["op"] == "prefill":
        state["caches"][0].prefill_compress(state["q"], state["k"], state["v"], state["prompt_len"], state["n"])
    elif state["case"]["graph"]:
        state["graph"].replay()
    else:
        _token(state, state["at"], 0)
        state["at"] = (state["at"] + 1) % state["tokens"]
    r = {"caches": [(c.k_cache, c.v_cache, c.codes_storage, c.scores, c.pos, c.fill, c.next_pos) for c in state["caches"]]}
    if state["case"]["op"] == "decode":
        r.update(victim=state["victim"], evicted=state["evicted"], out=state["out"])
    return r


def work(case):
    e, d, g, bits, h = 4 if case["dtype"] == "f32" else 2, case["dim"], case["group"], case["bits"], case["kv_heads"]
    budgets, lens = _lengths(case)
    if case["op"] == "prefill":
        # every key row and every evicting token's query rows once, the kept K / V rows in (K is in already) and out, the tables out
        n, kept = int(lens.sum()), int(torch.minimum(lens, budgets).sum())
        late = n - kept
        return {"bytes": h * (n * d * e + late * g * d * e + 3 * kept * d * e + kept * (bits / 8 + 8)) + d * bits * 4,
                "flops": h * 2 * d * bits * (n + late * g)}
    # a step: its q, k, v rows in, the code table in, the scores out, one slot rewritten; the attention: K and V of the budget in
    slots, units = int(budgets.sum()) * h, case["batch"] * h
    nbytes = units * ((g + 2) * d * e + 2 * d * e + bits / 8 + 12) + slots * (bits / 8 + 4) + d * bits * 4
    flops = units * (g + 1) * 2 * d * bits
    if case["attend"]:
        nbytes += slots * 2 * d * e + units * g * d * 4
        flops += slots * g * 4 * d
    calls = case["layers"] * case["tokens"]
    return {"bytes": calls * nbytes, "flops": calls * flops}


def tolerance(case):
    # codes, distances (whole numbers stored in fp32), victims, positions and the copied K / V rows are exact; only the
    # attention output is a sum of rounded fp32 terms
    return {"rel": 1e-5} if case["op"] == "decode" and case["attend"] else "exact"
