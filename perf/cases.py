"""The work that is timed: calls of the selective-KV path as a serving program makes them.

A case names one kind of call and its sizes.  The kinds, and what each stands for:

  prefill      every layer of a batch of prompts scored, selected and packed: HotPath.prefill
  layer        one layer of it, when that layer's KV cache is ready: HotPath.prefill_layer
  select_pack  selection and packing alone, on importances that are already there: HotPath.select_pack
  decode_step  one decode step, every layer's attention replayed from a CUDA graph, as a decode loop keeps it
  decode       one layer of a decode step, called directly: HotPath.decode
  two_lane     one layer of a decode step whose KV index is split by Algorithm 1, its remote entries fetched, all attended
  threshold    threshold selection under a cap and the packing of what it kept
  push         online transfer of the selected KV blocks of some layers, with the update of the KV mask

Head counts, head sizes, windows, prompt lengths, budgets and shares are those of `workloads.py` and of the tests:
8/2 heads of 64 (tiny), 32/8 of 128 (8B shape), 64/8 of 128 (70B shape).
"""
from __future__ import annotations

import math
import random

import torch

from paper_2607_28150_b200 import binding as sg
from paper_2607_28150_b200.pipeline import HotPath

NUM_BLOCKS = 1024          # KV blocks per layer of the online transfer
REMOTE_SHARE = 0.34        # on-demand share of the required entries
THRESHOLD_ALPHA = 5.0      # of scores with standard deviation 2


def _case(kind, layers, heads, window, batch, shortest, longest, keep, **more):
    """heads = (query heads, KV heads, head size); keep = selected share of each prompt."""
    hq, hkv, d = heads
    case = {"kind": kind, "layers": layers, "hq": hq, "hkv": hkv, "d": d, "window": window, "batch": batch,
            "shortest": shortest, "longest": longest, "lengths": 3, "keep": keep, "gathered": 0.0, "heavy": "scatter"}
    case.update(more)
    return case


def listed():
    tiny, small, large = (8, 2, 64), (32, 8, 128), (64, 8, 128)
    cases = {
        # the smallest call: one short prompt, a few KV heads; latency and launches are what it costs
        "prefill_tiny": _case("prefill", 1, tiny, 16, 1, 1024, 1024, 0.125),
        # a prefill engine that sends layer by layer: one layer of one 8K prompt
        "layer_8b": _case("layer", 1, small, 32, 1, 8192, 8192, 0.10),
        # the same for a ragged batch of long and short prompts with odd lengths
        "layer_ragged": _case("layer", 1, small, 32, 8, 2048, 32768, 0.10),
        # all layers of one 8K prompt at once
        "prefill_8b": _case("prefill", 32, small, 32, 1, 8192, 8192, 0.10),
        # long context: 32K tokens, 512 query rows per KV head, heavy keys in contiguous spans
        "prefill_70b": _case("prefill", 8, large, 64, 1, 32768, 32768, 0.0625, heavy="spans"),
        # selection and gather alone (importances come from elsewhere, or are profiled)
        "select_pack_8b": _case("select_pack", 32, small, 32, 1, 8192, 8192, 0.10),
        # decode loop at batch 1: 32 layers, two sources, latency-bound
        "decode_step_8b": _case("decode_step", 32, small, 32, 1, 8192, 8192, 0.10, gathered=0.34),
        # decode loop of a serving batch
        "decode_step_batch": _case("decode_step", 4, small, 32, 32, 4096, 4096, 0.20, gathered=0.25),
        # the largest attention call: everything required, half of it gathered
        "decode_full": _case("decode", 1, small, 32, 128, 4096, 4096, 1.0, gathered=0.5),
        # on-demand fetching of one layer for a ragged batch
        "two_lane_ragged": _case("two_lane", 1, small, 32, 8, 2048, 32768, 0.10),
        # the deployed rule: alpha and a maximum ratio, a different count per head
        "threshold_8b": _case("threshold", 32, small, 32, 1, 8192, 8192, 0.20),
        # online transfer of a few layers, two blocks of five selected
        "push_8b": _case("push", 8, small, 32, 1, 8192, 8192, 0.40),
    }
    return [dict(case, name=name) for name, case in cases.items()]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: any kind, sizes log-uniform, odd ones among them, no larger than the listed ones."""
    kind = rng.choice(("prefill", "layer", "prefill", "layer", "select_pack", "decode_step", "decode", "two_lane", "threshold", "push"))
    heads, window = rng.choice((((8, 2, 64), 16), ((32, 8, 128), 32), ((64, 8, 128), 64), ((32, 8, 128), rng.randint(12, 64)),
                                ((16, 8, 64), 32), ((32, 4, 128), rng.randint(8, 32))))
    hkv, rows = heads[1], heads[0] // heads[1] * window
    batch = 1 if rng.random() < 0.4 else _log_int(rng, 2, 96 if kind.startswith("decode") else 16)
    longest = _log_int(rng, 300, 32768 if batch <= 8 else 4096)
    shortest = longest if batch == 1 else max(64, _log_int(rng, max(64, longest // 16), longest))
    layers = 1 if kind in ("layer", "decode", "two_lane") else _log_int(rng, 1, 32)
    # the listed cases' largest: 2.1 M key rows (524 288 x 4 in a decode step), 512 query rows against all of them
    key_rows = batch * math.sqrt(shortest * longest) * hkv
    most = min(2.0e6, 1.0e9 / rows) if kind in ("prefill", "layer") else 2.0e6
    layers = max(1, min(layers, int(most / key_rows)))
    if kind.startswith("decode"):
        keep, gathered = rng.choice((0.05, 0.10, 0.20, 0.5, 1.0)), rng.choice((0.0, 0.25, 0.34, 0.5))
    else:
        keep, gathered = rng.choice((0.05, 0.10, 0.15, 0.20, 0.40)), 0.0
    return _case(kind, layers, heads, window, batch, shortest, longest, keep, gathered=gathered, lengths=rng.randrange(1 << 30),
                 heavy=rng.choice(("scatter", "spans")))


# ------------------------------------------------------------------------------------------------- sizes
def _lengths(case):
    rng = random.Random(case["lengths"])
    lo, hi = case["shortest"], case["longest"]
    if case["batch"] == 1 or lo == hi:
        return [hi] * case["batch"]
    return [rng.randint(lo, hi) for _ in range(case["batch"])]


def _required(case):
    """Required entries per KV head, per sequence (the budget of a selection)."""
    return [min(n, max(1, math.ceil(case["keep"] * n - 1e-9))) for n in _lengths(case)]


def _gathered(case):
    """How many of them a decode step reads through the local index."""
    return [min(k, int(round(case["gathered"] * k))) for k in _required(case)]


def work(case):
    L, hq, hkv, d, B, W = (case[k] for k in ("layers", "hq", "hkv", "d", "batch", "window"))
    T, K, NL = sum(_lengths(case)), sum(_required(case)), sum(_gathered(case))
    row, kind = 2 * d, case["kind"]                              # bytes of one K or V row
    q_out = 2 * B * hq * row + 4 * B * hq                        # query, output and log-sum-exp of one attention call
    attend = 4 * (hq // hkv) * d                                 # operations per attended entry and KV head
    if kind in ("prefill", "layer"):
        # K and the window queries in; importance, index and packed rows out; the selected V rows in
        by = L * (hkv * (T * row + 4 * T + K * (4 + 3 * row)) + B * W * hq * row)
        return {"bytes": by, "flops": 2 * L * hq * W * T * d}
    if kind == "select_pack":
        return {"bytes": L * hkv * (4 * T + K * (4 + 4 * row)), "flops": 0}
    if kind in ("decode_step", "decode"):
        return {"bytes": L * (hkv * (2 * K * row + 4 * NL) + q_out), "flops": L * hkv * K * attend}
    if kind == "two_lane":
        # index and mask in; reordered row, local and remote lists out; the remote rows in and out; all entries attended
        remote = REMOTE_SHARE * K
        return {"bytes": hkv * (12 * K + 4 * remote * row + 2 * (K - remote) * row) + T + q_out, "flops": hkv * K * attend}
    if kind == "threshold":
        # the scores in, the index out, the kept rows in and out; what passes is estimated from the expected maximum
        kept = 0.0
        for n, cap in zip(_lengths(case), _required(case)):
            a = math.sqrt(2.0 * math.log(n))
            top = a - (math.log(math.log(n)) + math.log(4.0 * math.pi)) / (2.0 * a)
            kept += min(cap, n * 0.5 * math.erfc((top - THRESHOLD_ALPHA / 2.0) / math.sqrt(2.0)))
        return {"bytes": L * hkv * (4 * T + 4 * K + 4 * kept * row), "flops": 0}
    return {"bytes": L * case["keep"] * T * (4 * hkv * row + 1), "flops": 0}


def tolerance(case):
    kind = case["kind"]
    if kind in ("select_pack", "threshold", "push"):
        return "exact"
    if kind in ("prefill", "layer"):
        # importances are fp32 sums of exponentials of fp32 scores (measured against 64-bit arithmetic on the same inputs:
        # relative error 2.5e-7, largest 1.5e-6); an index entry may differ where two importances are that close, and then
        # shifts the entries and packed rows behind it
        return {"rel": 1e-6, "max": 8e-6, "differ": 0.01}
    # outputs are bf16 and probabilities are rounded to bf16 (measured against 64-bit attention over the same rows:
    # relative error 2.2e-3, largest 7.8e-3)
    return {"rel": 8e-3, "max": 0.03}


# ------------------------------------------------------------------------------------------------- inputs
def _unit(x):
    return x / x.norm(dim=-1, keepdim=True).clamp_min(1e-30)


def _heavy_positions(case, n, gen):
    """Sinks and heavy keys of one prompt: 1 % of the tokens, or four spans of 256."""
    lo, hi = 4, max(5, n - case["window"])
    if case["heavy"] == "spans" and (hi - lo) // 256 >= 4:
        starts = lo + 256 * torch.randperm((hi - lo) // 256, generator=gen, device="cuda")[:4]
        pos = (starts[:, None] + torch.arange(256, device="cuda")).reshape(-1)
    else:
        pos = lo + torch.randperm(hi - lo, generator=gen, device="cuda")[: max(1, n // 100)]
    return torch.cat([torch.arange(min(4, n), device="cuda"), pos]).clamp_max(n - 1)


def _normal(gen, *shape):
    return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.bfloat16)


def _caches(case, gen):
    """Window queries and K / V caches of all layers: normal values, with sinks and heavy keys along the mean query."""
    L, hq, hkv, d, W = (case[k] for k in ("layers", "hq", "hkv", "d", "window"))
    lens = _lengths(case)
    T = sum(lens)
    q = _normal(gen, L, len(lens), W, hq, d)
    k, v = _normal(gen, L, T, hkv, d), _normal(gen, L, T, hkv, d)
    at = 0
    for b, n in enumerate(lens):
        u = _unit(q[:, b].float().reshape(L, W, hkv, hq // hkv, d).mean(dim=(1, 3)))[:, None]
        pos = at + _heavy_positions(case, n, gen)
        k[:, pos] = (4.0 * math.sqrt(d) * _unit(0.9 * u + 0.436 * _unit(k[:, pos].float()))).bfloat16()
        at += n
    return q, k, v


def _positions(case, counts, gen):
    """Per layer, KV head and sequence `counts[b]` distinct positions in random order: int32 [L][H_kv][sum counts]."""
    rows, parts = case["layers"] * case["hkv"], []
    for n, c in zip(_lengths(case), counts):
        parts.append(torch.rand(rows, n, generator=gen, device="cuda").argsort(dim=1)[:, :c].int())
    return torch.cat(parts, dim=1).reshape(case["layers"], case["hkv"], -1).contiguous()


def _prefix(counts):
    return torch.tensor([sum(counts[:i]) for i in range(len(counts) + 1)], dtype=torch.int32, device="cuda")


def _hot_path(case, budgets):
    return HotPath(case["layers"], case["hq"], case["hkv"], case["d"], case["window"], _lengths(case), budgets)


def _importance_like(case, gen):
    """Importances as scoring gives them: softmax mass, most tokens within a few octaves, a few far above."""
    x = torch.randn(case["layers"], case["hkv"], sum(_lengths(case)), generator=gen, device="cuda")
    heavy = torch.rand(x.shape, generator=gen, device="cuda") < 0.01
    return torch.exp(0.7 * x + 4.0 * heavy)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed * 1000003 + 17)
    kind, lens, need = case["kind"], _lengths(case), _required(case)
    L, hq, hkv, d, B = (case[k] for k in ("layers", "hq", "hkv", "d", "batch"))
    state = {"kind": kind}
    if kind in ("prefill", "layer"):
        q, k, v = _caches(case, gen)
        state.update(hp=_hot_path(case, need), q=q, k=k, v=v)
    elif kind == "select_pack":
        hp = _hot_path(case, need)
        hp.importance.copy_(_importance_like(case, gen))
        state.update(hp=hp, k=_normal(gen, L, sum(lens), hkv, d), v=_normal(gen, L, sum(lens), hkv, d))
    elif kind in ("decode_step", "decode"):
        loc = _gathered(case)
        hp = _hot_path(case, [n - m for n, m in zip(need, loc)])
        hp.packed_k.copy_(_normal(gen, *hp.packed_k.shape).view(torch.int16))
        hp.packed_v.copy_(_normal(gen, *hp.packed_v.shape).view(torch.int16))
        state.update(hp=hp, k=_normal(gen, L, sum(lens), hkv, d), v=_normal(gen, L, sum(lens), hkv, d),
                     q=_normal(gen, L, B, hq, d), idx=_positions(case, loc, gen), cu_nloc=_prefix(loc), nloc=sum(loc),
                     out=torch.zeros(L, B, hq, d, dtype=torch.bfloat16, device="cuda"),
                     lse=torch.zeros(L, B, hq, device="cuda"))
        if kind == "decode_step":
            _attend(state)                                       # once outside the graph: the workspaces are made here
            torch.cuda.synchronize()
            state["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(state["graph"]):
                _attend(state)
    elif kind == "two_lane":
        hp = _hot_path(case, need)
        at = torch.repeat_interleave(torch.arange(B, device="cuda"), torch.tensor(need, device="cuda"))
        index = _positions(case, need, gen)[0] + (at * (1 << 20)).int()      # sorted inside each sequence
        hp.sel_idx[0].copy_(index.sort(dim=1).values & ((1 << 20) - 1))
        mask = torch.where(torch.rand(sum(lens), generator=gen, device="cuda") < REMOTE_SHARE, 2, 1).to(torch.int8)
        hp.packed_k.zero_(), hp.packed_v.zero_()
        state.update(hp=hp, mask=mask, k=_normal(gen, 1, sum(lens), hkv, d)[0], v=_normal(gen, 1, sum(lens), hkv, d)[0],
                     q=_normal(gen, B, hq, d), out=torch.zeros(B, hq, d, dtype=torch.bfloat16, device="cuda"),
                     lse=torch.zeros(B, hq, device="cuda"),
                     lists=[torch.zeros_like(hp.sel_idx[0]) for _ in range(3)],
                     counts=[torch.zeros(B, hkv, dtype=torch.int32, device="cuda") for _ in range(2)])
    elif kind == "threshold":
        hp = _hot_path(case, need)                               # the caps
        hp.packed_k.zero_(), hp.packed_v.zero_()
        scores = 2.0 * torch.randn(L, hkv, sum(lens), generator=gen, device="cuda")
        state.update(hp=hp, scores=scores, counts=torch.zeros(L, B, hkv, dtype=torch.int32, device="cuda"),
                     k=_normal(gen, L, sum(lens), hkv, d), v=_normal(gen, L, sum(lens), hkv, d))
    else:
        hp = _hot_path(case, need)
        chosen = torch.rand(L * NUM_BLOCKS, generator=gen, device="cuda") < case["keep"]
        k, v = _normal(gen, L, sum(lens), hkv, d), _normal(gen, L, sum(lens), hkv, d)
        state.update(hp=hp, chosen=chosen.nonzero()[:, 0].int(), k=k, v=v, dst_k=torch.zeros_like(k), dst_v=torch.zeros_like(v),
                     mask=torch.full((L, sum(lens)), 2, dtype=torch.int8, device="cuda"))
    return state


# ------------------------------------------------------------------------------------------------- one pass
def _attend(s):
    hp = s["hp"]
    for layer in range(hp.L):
        hp.decode(layer, s["q"][layer], s["k"][layer], s["v"][layer], s["idx"][layer], s["cu_nloc"], s["nloc"], s["out"][layer],
                  s["lse"][layer])


def run(s):
    kind, hp = s["kind"], s["hp"]
    if kind == "prefill":
        hp.prefill(s["q"], s["k"], s["v"])
        return [hp.importance, hp.sel_idx, hp.packed_k, hp.packed_v]
    if kind == "layer":
        hp.prefill_layer(0, s["q"], s["k"], s["v"])
        return [hp.importance, hp.sel_idx, hp.packed_k, hp.packed_v]
    if kind == "select_pack":
        hp.select_pack(s["k"], s["v"])
        return [hp.sel_idx, hp.packed_k, hp.packed_v]
    if kind == "decode_step":
        s["graph"].replay()
        return [s["out"], s["lse"]]
    if kind == "decode":
        _attend(s)
        return [s["out"], s["lse"]]
    if kind == "two_lane":
        reordered, local, remote = s["lists"]
        n_local, n_remote = s["counts"]
        sg.sg_split_index(hp.shape1, hp.sel_idx[0], hp.cu_k, hp.K_tot, s["mask"], True, reordered, local, remote, n_local, n_remote,
                          hp.status)
        sg.sg_pack_kv_counted(hp.shape1, s["k"], s["v"], reordered, hp.cu_k, hp.K_tot, n_remote, hp.packed_k[0], hp.packed_v[0],
                              hp.status)
        sg.sg_sparse_decode_attn_counted(hp.shape1, s["q"], hp.packed_k[0], hp.packed_v[0], hp.cu_k, hp.K_tot, n_remote, s["k"], s["v"],
                                         reordered, hp.cu_k, hp.K_tot, s["out"], s["lse"], 0.0, hp.status, None, n_remote)
        return [s["out"], s["lse"], reordered, n_local, n_remote, hp.packed_k, hp.packed_v]
    if kind == "threshold":
        sg.sg_select_threshold(hp.shape, s["scores"], THRESHOLD_ALPHA, hp.cu_k, hp.K_tot, hp.sel_idx, s["counts"], hp.status)
        sg.sg_pack_kv_counted(hp.shape, s["k"], s["v"], hp.sel_idx, hp.cu_k, hp.K_tot, s["counts"], hp.packed_k, hp.packed_v, hp.status)
        return [hp.sel_idx, s["counts"], hp.packed_k, hp.packed_v]
    sg.sg_push_blocks(hp.shape, NUM_BLOCKS, 0, s["chosen"], s["k"], s["v"], s["dst_k"], s["dst_v"], s["mask"])
    return [s["dst_k"], s["dst_v"], s["mask"]]
