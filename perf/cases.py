"""Timed cases of the speculative-step hot path: what a decode loop asks of the library.

A case is one of five kinds of pass, all through the public binding:

  step        a whole speculative step: draft-tree expansion, tree attention on every layer, greedy
              verification, KV-cache compaction.  `graph` says how a serving program runs it: replayed
              from a captured CUDA graph, or called eagerly from Python between the layers of a model.
  sampled     the vocabulary side of a step at temperature > 0: tree expansion and acceptance under sampling.
  level       the level form of the expansion (a draft model runs between the levels), called eagerly.
  controller  one call of the action controller, the policy asked every `interval` steps.
  shard       one rank's calls of a step whose vocabulary is split over several GPUs (the all-gathers
              between them are the caller's).

Shapes are those of the repository's five workloads (`synth.WORKLOADS`) and generic ones around them.
Logits are fp32 Gumbel noise with one peak of probability 0.7 per row; the target agrees with a tree
node's first child with probability 0.8; Q, K and V are bf16 N(0, 1).
"""
import math
import random

import numpy as np
import torch

from paper_2601_12212_b200 import binding, synth

P_AGREE = 0.8
PEAK = 0.7


def _step(name, batch, hq, hkv, dim, vocab, layers, prefix, tt, d, k, graph, prefix_hi=0):
    return {"name": name, "kind": "step", "batch": batch, "hq": hq, "hkv": hkv, "dim": dim, "vocab": vocab,
            "layers": layers, "prefix": prefix, "prefix_hi": prefix_hi or prefix, "tt": tt, "d": d, "k": k,
            "graph": graph}


def listed():
    return [
        # The smallest step (workload 1), called from Python: nothing but latency and launches.
        _step("step tiny", 1, 4, 1, 64, 1024, 1, 128, 16, 4, 4, False),
        # The configuration the repository's metric is quoted on (workload 2): single-user decoding.
        _step("step 8b graph", 1, 32, 8, 128, 128256, 32, 1024, 60, 7, 10, True),
        # The largest tree of the paper's action space on the same model, its layers run eagerly.
        _step("step 8b wide eager", 1, 32, 8, 128, 128256, 32, 2048, 128, 8, 32, False),
        # A model without grouped heads (workload 3), a mid-sized tree of its grid.
        _step("step 13b graph", 1, 40, 40, 128, 32000, 40, 2048, 48, 6, 8, True),
        # The largest model (workload 4).
        _step("step 70b graph", 1, 64, 8, 128, 128256, 80, 4096, 96, 8, 12, True),
        # Serving a ragged batch, every sequence with its own tree and prefix (workload 5).
        _step("step ragged 8 graph", 8, 32, 8, 128, 128256, 32, 1024, 80, 8, 12, True, prefix_hi=8192),
        # A vocabulary with one added token (rows that are not 16-byte aligned), 7 heads per KV head, odd
        # prefixes, two users, eager.
        _step("step odd eager", 2, 28, 4, 128, 32001, 28, 777, 47, 5, 7, False, prefix_hi=1531),
        # One user with a long document: attention over the prefix is what there is.
        _step("step long graph", 1, 32, 8, 128, 128256, 32, 32000, 32, 4, 8, True),
        # Sampling at temperature 1 on workload 2's tree.
        {"name": "sampled 8b", "kind": "sampled", "batch": 1, "vocab": 128256, "tt": 60, "d": 7, "k": 10,
         "temperature": 1.0},
        # A draft model that runs between the levels, workload 2's tree.
        {"name": "level 8b", "kind": "level", "batch": 1, "vocab": 128256, "tt": 60, "d": 7, "k": 10},
        # The controller of eight sequences: three hidden states of width 4096, the paper's 180 actions.
        {"name": "controller 8", "kind": "controller", "batch": 8, "width": 4096, "hidden": 128, "interval": 4,
         "temperature": 1.0},
        # One of four ranks of workload 4, which the paper runs on four GPUs.
        {"name": "shard 70b 4 ranks", "kind": "shard", "batch": 1, "vocab": 128256, "ranks": 4, "tt": 96, "d": 8,
         "k": 12},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_vocab(rng):
    # sizes as they come: mostly multiples of 64, some with a few tokens added
    v = _log(rng, 1000, 152000)
    return v if rng.random() < 0.35 else (v + 63) // 64 * 64


def _draw_one(rng):
    kind = rng.choice(["step"] * 8 + ["sampled", "level", "controller", "shard"])
    tt, d, k = rng.randint(4, 128), rng.randint(2, 8), rng.choice([rng.randint(2, 12), rng.randint(4, 32)])
    batch = _log(rng, 1, 16)
    if kind == "controller":
        return {"kind": kind, "batch": batch, "width": _log(rng, 512, 8192), "hidden": rng.choice([64, 128, 256]),
                "interval": rng.randint(1, 10), "temperature": rng.choice([0.0, 1.0])}
    vocab = _draw_vocab(rng)
    if kind != "step":
        c = {"kind": kind, "batch": batch, "vocab": vocab, "tt": tt, "d": d, "k": k}
        if kind == "sampled":
            c["temperature"] = rng.choice([0.5, 0.7, 1.0])
        if kind == "shard":
            c["ranks"] = rng.choice([2, 4, 8])
            c["vocab"] = max(vocab, 64 * c["ranks"])
        return c
    hkv = rng.choice([1, 2, 4, 8, 8, 10, 16, 32, 40])
    group = rng.choice([1, 2, 4, 4, 5, 7, 8]) if hkv <= 10 else rng.choice([1, 2])
    lo = _log(rng, 64, 32000)
    hi = min(32000, _log(rng, lo, 8 * lo)) if batch > 1 else lo
    c = _step("", batch, hkv * group, hkv, rng.choice([64, 128, 128]), vocab, _log(rng, 1, 80), lo, tt, d, k,
              rng.random() < 0.6, prefix_hi=hi)
    del c["name"]
    return c


def draw(rng):
    most = [work(c) for c in listed()]
    limit = max(max(w["bytes"], w["flops"] / 200) for w in most)
    while True:
        c = _draw_one(rng)
        w = work(c)
        held = 4 * c.get("vocab", 0) * c["batch"] * (c.get("d", 0) * c.get("k", 0) + c.get("tt", 0))
        if c["kind"] == "step":
            held += 4 * c["layers"] * c["batch"] * (_capacity(c) * c["hkv"] + c["tt"] * c["hq"]) * c["dim"]
        if max(w["bytes"], w["flops"] / 200) <= limit and held <= 12e9:
            return c


def _sequences(case):
    """(TT, d, k, prefix) of every sequence: the case's own for one sequence; in a batch every sequence has
    its own action (up to the case's limits, which the first one takes) and prefix, as in a ragged batch."""
    mix = random.Random(17)
    n, lo, hi = case["batch"], case.get("prefix", 0), case.get("prefix_hi", 0)
    out = []
    for b in range(n):
        f = [1.0, 1.0, 1.0] if b == 0 else [mix.random() for _ in range(3)]
        out.append((max(2, round(case["tt"] * (0.2 + 0.8 * f[0]))), max(1, round(case["d"] * (0.4 + 0.6 * f[1]))),
                    max(1, round(case["k"] * (0.35 + 0.65 * f[2]))),
                    lo + (hi - lo) * ((5 * b + 3) % n) // max(1, n - 1)))
    return out


def _nodes(tt, d, k):
    return min(tt, 1 + k + (d - 1) * k * k)


def _capacity(case):
    return (case["prefix_hi"] + case["tt"] + 63) // 64 * 64


def work(case):
    if case["kind"] == "controller":
        f = 3 * case["width"]
        n_act = len(synth.action_space())
        # the policy is asked at one step in `interval`: its weights once, the states of every sequence
        weights = case["hidden"] * (f + case["hidden"] + n_act)
        return {"bytes": (4 * weights + 2 * f * case["batch"]) / case["interval"] + 64 * case["batch"],
                "flops": 2 * weights * case["batch"] / case["interval"]}
    nbytes = flops = 0
    share = 1.0 / case.get("ranks", 1)
    for tt, d, k, prefix in _sequences(case):
        n = _nodes(tt, d, k)
        nbytes += 4 * case["vocab"] * (1 + (d - 1) * k) * share  # every draft row once
        if case["kind"] in ("step", "shard"):
            nbytes += 4 * case["vocab"] * n * share  # every node's target row once
        elif case["kind"] == "sampled":
            nbytes += 8 * case["vocab"]  # at least the root's target and draft row
        if case["kind"] == "step":
            kv, q = 2 * (prefix + n) * case["hkv"] * case["dim"] * 2, n * case["hq"] * case["dim"] * 2
            nbytes += case["layers"] * (kv + 2 * q)
            flops += case["layers"] * 4 * n * case["hq"] * (prefix + n) * case["dim"]
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["kind"] == "step":
        return {"rel": 5e-3, "max": 2e-2}  # attention output in bf16; everything else is whole numbers
    if case["kind"] in ("level", "shard"):
        return {"rel": 1e-6, "max": 1e-5}  # log-probabilities over fp32 partial sums
    if case["kind"] == "controller":
        return {"rel": 2e-5, "max": 2e-4}  # fp32 sums of 3 x width terms
    return "exact"


class State:
    """What a decode loop keeps: the context, the step parameters, the inputs and the output buffers."""


def _i32(*shape, fill=0):
    return torch.full(shape, fill, dtype=torch.int32, device="cuda")


def _peaked(gen, rows, vocab, peak=None):
    """fp32 [rows][vocab]: Gumbel(0, 1) noise and one entry per row (drawn, or given) of probability PEAK."""
    x = torch.rand(rows, vocab, generator=gen, device="cuda").clamp_(1e-7, 1 - 1e-7).log_().neg_().log_().neg_()
    if peak is None:
        peak = torch.randint(vocab, (rows,), generator=gen, device="cuda")
    peak = peak.view(rows, 1)
    x.scatter_(1, peak, float("-inf"))
    return x.scatter_(1, peak, x.logsumexp(1, keepdim=True) + math.log(PEAK / (1 - PEAK)))


def _trees(s, case, gen, vocab, own_vocab=None):
    """Context (for `own_vocab` columns where a rank holds a part of the vocabulary), step parameters, draft
    rows and the tree's output buffers."""
    B, T, MD, MK = case["batch"], case["tt"], case["d"], case["k"]
    s.case, s.B, s.T, s.MD, s.MK, s.V = case, B, T, MD, MK, own_vocab or vocab
    s.ctx = binding.Context(case.get("hq", 8), case.get("hkv", 2), case.get("dim", 128), s.V, max_batch=B, max_tt=T,
                            max_k=MK, max_depth=MD)
    s.steps = torch.tensor(_sequences(case), dtype=torch.int32, device="cuda")
    s.steps_next = torch.zeros_like(s.steps)
    s.root = torch.randint(vocab, (B,), generator=gen, device="cuda", dtype=torch.int32)
    s.draft = torch.cat([_peaked(gen, MD * MK, vocab).view(1, MD, MK, vocab) for _ in range(B)])
    s.tree = {"tokens": _i32(B, T), "parent": _i32(B, T), "depth": _i32(B, T), "position_ids": _i32(B, T),
              "mask": torch.zeros(B, T, 2, dtype=torch.int64, device="cuda"), "retrieve": _i32(B, T, MD + 1),
              "n_leaves": _i32(B), "n_nodes": _i32(B)}
    s.accept = {"argmax": _i32(B, T), "path": _i32(B, MD + 1), "length": _i32(B), "tokens": _i32(B, MD + 1)}


def _expand(s):
    t = s.tree
    binding.resps_tree_expand(s.ctx, s.steps, s.B, s.draft, s.MD * s.MK * s.V, s.MK * s.V, s.V, s.MD, s.MK, s.root,
                              t["tokens"], t["parent"], t["depth"], t["position_ids"], t["mask"], t["retrieve"],
                              t["n_leaves"], t["n_nodes"])


def _target(s, gen, seed, vocab):
    """Target rows of the tree in `s.tree`: with probability P_AGREE a node's peak is its first child's token."""
    rng = np.random.default_rng(seed)
    tok, par, num = (s.tree[n].cpu().numpy() for n in ("tokens", "parent", "n_nodes"))
    peak, agree = rng.integers(0, vocab, (s.B, s.T)), rng.random((s.B, s.T)) < P_AGREE
    for b in range(s.B):
        for c in range(int(num[b]) - 1, 0, -1):  # the first child is written last
            if agree[b, par[b, c]]:
                peak[b, par[b, c]] = tok[b, c]
    peak = torch.from_numpy(peak).cuda()
    return torch.cat([_peaked(gen, s.T, vocab, peak[b]).view(1, s.T, vocab) for b in range(s.B)])


def _prepare_step(s, case, gen, seed):
    _trees(s, case, gen, case["vocab"])
    _expand(s)
    s.target = _target(s, gen, seed, case["vocab"])
    B, NL, hq, hkv, D, cap = s.B, case["layers"], case["hq"], case["hkv"], case["dim"], _capacity(case)
    bf = dict(generator=gen, device="cuda", dtype=torch.bfloat16)
    s.q = torch.randn(NL, B, s.T, hq, D, **bf)
    s.o = torch.zeros_like(s.q)
    s.k, s.v = torch.randn(NL, B, hkv, cap, D, **bf), torch.randn(NL, B, hkv, cap, D, **bf)
    # the layers' buffers, as a model holds them
    s.layers = list(zip(s.q.unbind(0), s.o.unbind(0), s.k.unbind(0), s.v.unbind(0)))
    s.k_ptrs, s.v_ptrs = (binding.layer_pointer_table(list(c.unbind(0))) for c in (s.k, s.v))
    s.strides, s.cap, s.scale = (hkv * cap * D, cap * D, D), cap, 1.0 / math.sqrt(D)
    s.out = {"tree": s.tree, "accept": s.accept, "steps": s.steps_next, "o": s.o, "k": s.k, "v": s.v}
    s.graph = None
    if case["graph"]:
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            _step_calls(s)
        s.graph = graph


def _step_calls(s):
    t, a = s.tree, s.accept
    _expand(s)
    for q, o, k, v in s.layers:
        binding.resps_tree_attention(s.ctx, s.steps, t["n_nodes"], s.B, q, o, None, k, v, *s.strides, s.cap,
                                     t["mask"], s.scale)
    binding.resps_verify_accept(s.ctx, s.steps, t["n_nodes"], s.B, s.target, s.T * s.V, s.V, t["tokens"], t["parent"],
                                a["argmax"], a["path"], a["length"], a["tokens"], s.steps_next)
    binding.resps_kv_compact(s.ctx, s.steps, s.B, a["path"], a["length"], s.k_ptrs, s.v_ptrs, len(s.layers),
                             *s.strides, s.cap)


def _run_step(s):
    if s.graph is not None:
        s.graph.replay()
    else:
        _step_calls(s)
    return s.out


def _prepare_sampled(s, case, gen, seed):
    _trees(s, case, gen, case["vocab"])
    _expand(s)
    s.target = _target(s, gen, seed, case["vocab"])
    u = dict(generator=gen, device="cuda", dtype=torch.float64)
    s.u_accept, s.u_sample = torch.rand(s.B, s.MD + 1, s.MK, **u), torch.rand(s.B, s.MD + 1, **u)
    s.accept.pop("argmax")
    s.out = {"tree": s.tree, "accept": s.accept, "steps": s.steps_next}


def _run_sampled(s):
    t, a, V = s.tree, s.accept, s.V
    _expand(s)
    binding.resps_verify_accept_sampled(s.ctx, s.steps, t["n_nodes"], s.B, s.target, s.T * V, V, s.draft,
                                        s.MD * s.MK * V, s.MK * V, V, s.case["temperature"], t["tokens"], t["parent"],
                                        s.u_accept, s.u_sample, a["path"], a["length"], a["tokens"], s.steps_next)
    return s.out


def _prepare_level(s, case, gen, seed):
    _trees(s, case, gen, case["vocab"])
    B, MK = s.B, s.MK
    # a draft model writes each level's rows into a buffer of their own
    s.rows = [s.draft[:, j].contiguous() for j in range(s.MD)]
    s.draft = None
    s.frontier = [{"tokens": _i32(B, MK), "parent_slot": _i32(B, MK), "position_ids": _i32(B, MK),
                   "node_index": _i32(B, MK), "mask": torch.zeros(B, MK, 2, dtype=torch.int64, device="cuda"),
                   "score": torch.zeros(B, MK, dtype=torch.float64, device="cuda")} for _ in range(s.MD)]
    # one tensor per array over the levels
    s.out = {n: torch.stack([f[n] for f in s.frontier]) for n in s.frontier[0]}
    s.frontier = [{n: s.out[n][j] for n in s.out} for j in range(s.MD)]
    s.out["tree"] = s.tree


def _run_level(s):
    t = s.tree
    binding.resps_tree_expand_begin(s.ctx, s.steps, s.B, s.MK)
    for j, (rows, f) in enumerate(zip(s.rows, s.frontier)):
        binding.resps_tree_expand_level(s.ctx, s.steps, s.B, j, rows, s.MK * s.V, s.V, f["tokens"], f["parent_slot"],
                                        f["position_ids"], f["node_index"], f["mask"], f["score"])
    binding.resps_tree_expand_finish(s.ctx, s.steps, s.B, s.root, t["tokens"], t["parent"], t["depth"],
                                     t["position_ids"], t["mask"], t["retrieve"], t["n_leaves"], t["n_nodes"])
    return s.out


def _prepare_controller(s, case, gen, seed):
    B, W, H = case["batch"], case["width"], case["hidden"]
    actions = torch.tensor(synth.action_space(), dtype=torch.int32, device="cuda")
    A, F = len(actions), 3 * W
    s.case, s.B = case, B
    s.ctx = binding.Context(8, 2, 128, 1000, max_batch=B, max_tt=128, max_k=32, max_depth=8)
    r = dict(generator=gen, device="cuda")
    s.weights = [torch.randn(H, F, **r) / math.sqrt(F), 0.1 * torch.randn(H, **r), torch.randn(H, H, **r) / math.sqrt(H),
                 0.1 * torch.randn(H, **r), 0.5 * torch.randn(A, H, **r), 0.1 * torch.randn(A, **r), actions]
    s.policy = binding.make_policy(*s.weights)
    s.hidden = [torch.randn(B, W, dtype=torch.bfloat16, **r) for _ in range(3)]
    s.uniform = torch.rand(B, dtype=torch.float64, **r)
    s.accepted = torch.randint(7, (B,), dtype=torch.int32, **r)
    s.seconds = 4e-4 + 5e-4 * torch.rand(B, **r)
    s.out = {"state": _i32(B, 4), "steps": torch.tensor([[1, 1, 1, 100 + b] for b in range(B)], dtype=torch.int32,
                                                        device="cuda"),
             "reward": torch.zeros(B, device="cuda"), "logits": torch.zeros(B, A, device="cuda"), "action": _i32(B)}


def _run_controller(s):
    o = s.out
    binding.resps_controller_step(s.ctx, s.policy, *s.hidden, s.case["width"], s.B, s.case["interval"],
                                  s.case["temperature"], s.uniform, s.accepted, s.seconds, o["state"], o["steps"],
                                  o["reward"], o["logits"], o["action"])
    return o


def _prepare_shard(s, case, gen, seed):
    P, vocab = case["ranks"], case["vocab"]
    cols = binding.shard_columns(vocab, P)
    _trees(s, case, gen, vocab, own_vocab=cols[0][1])
    B, T, MK = s.B, s.T, s.MK
    ctxs = [s.ctx] + [binding.Context(8, 2, 128, wd, max_batch=B, max_tt=T, max_k=MK, max_depth=s.MD)
                      for _, wd in cols[1:]]
    rows = int(binding.load().resps_scan_rows(s.ctx.handle))
    s.offset = torch.tensor([off for off, _ in cols], dtype=torch.int32, device="cuda")
    # what the all-gathers deliver; this rank's calls write their own slice in place
    s.all_val, s.all_id = torch.zeros(P, B, rows, MK, device="cuda"), _i32(P, B, rows, MK)
    s.all_lse = torch.zeros(P, B, rows, dtype=torch.float64, device="cuda")
    s.all_key = torch.zeros(P, B, T, dtype=torch.int64, device="cuda")
    own = [s.draft[..., off:off + wd].contiguous() for off, wd in cols]
    s.draft = own[0]
    for p in range(P):
        _scan_shard(s, ctxs[p], own[p], p)
    _expand_merge(s)
    target = _target(s, gen, seed, vocab)
    own = [target[..., off:off + wd].contiguous() for off, wd in cols]
    s.target = own[0]
    for p in range(P):
        _argmax_shard(s, ctxs[p], own[p], p)
    torch.cuda.synchronize()
    for c in ctxs[1:]:
        c.close()
    s.out = {"tree": s.tree, "accept": s.accept, "steps": s.steps_next, "val": s.all_val[0], "id": s.all_id[0],
             "lse": s.all_lse[0], "key": s.all_key[0]}


def _scan_shard(s, ctx, rows, p):
    V = rows.shape[-1]
    binding.resps_row_scan_shard(ctx, s.steps, s.B, rows, s.MD * s.MK * V, s.MK * V, V, s.MD, s.MK, s.all_val[p],
                                 s.all_id[p], s.all_lse[p])


def _expand_merge(s):
    t = s.tree
    binding.resps_tree_expand_merge(s.ctx, s.steps, s.B, s.MD, s.MK, s.case["ranks"], s.all_val, s.all_id, s.all_lse,
                                    s.offset, s.root, t["tokens"], t["parent"], t["depth"], t["position_ids"],
                                    t["mask"], t["retrieve"], t["n_leaves"], t["n_nodes"])


def _argmax_shard(s, ctx, rows, p):
    V = rows.shape[-1]
    binding.resps_target_argmax_shard(ctx, s.tree["n_nodes"], s.B, rows, s.T * V, V, s.all_key[p])


def _run_shard(s):
    t, a = s.tree, s.accept
    _scan_shard(s, s.ctx, s.draft, 0)
    _expand_merge(s)
    _argmax_shard(s, s.ctx, s.target, 0)
    binding.resps_verify_accept_merge(s.ctx, s.steps, t["n_nodes"], s.B, s.case["ranks"], s.all_key, s.offset,
                                      t["tokens"], t["parent"], a["argmax"], a["path"], a["length"], a["tokens"],
                                      s.steps_next)
    return s.out


_KINDS = {"step": (_prepare_step, _run_step), "sampled": (_prepare_sampled, _run_sampled),
          "level": (_prepare_level, _run_level), "controller": (_prepare_controller, _run_controller),
          "shard": (_prepare_shard, _run_shard)}


def prepare(case, seed):
    s = State()
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    _KINDS[case["kind"]][0](s, case, gen, seed)
    return s


def run(state):
    return _KINDS[state.case["kind"]][1](state)
