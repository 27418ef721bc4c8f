"""Timed cases of the library: what a serving program has it do in one speculative cycle.

Every case goes through the public binding.  A case names the part of the cycle it times:

  step     tree convolution + tree scan of every node, then the commit of the accepted path (one or more layers)
  fused    the same cycle through ``commit_verify``: the previous commit folded into this verify
  cached   a verify that exports every node's state beside the outputs (state caching instead of recomputation)
  attn     the full-attention layer of the cycle: KV write, tree attention, KV publication
  accept   the acceptance walk over full-vocabulary target (and proposal) rows
  select   the draft selection over full-vocabulary logits

Sizes are those of the benchmark configurations and of the tests, and whatever lies between them.
"""
from __future__ import annotations

import math
import random
from typing import Dict, List

import numpy as np
import torch

from paper_2609_23900_b200 import binding

_DT = {"f32": torch.float32, "bf16": torch.bfloat16}
_P_STOP = 0.35       # accepted lengths: P(L = l) = p (1 - p)^(l - 1), cut at the leaf
_SPINE = 12          # longest principal chain of a "spine" tree
_CHAIN = 16          # length of the chains of a "chains" tree

_shared: Dict[int, binding.Context] = {}


def _ctx() -> binding.Context:
    """One context per device, kept for the life of the process, as a server keeps it."""
    dev = torch.cuda.current_device()
    if dev not in _shared:
        _shared[dev] = binding.Context(dev)
    return _shared[dev]


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _gdn(kind, B, N, L, shape, depth, **kw):
    c = dict(kind=kind, B=B, N=N, rows=N, L=L, shape=shape, depth=depth, Hk=16, Hv=32, d=128, dtype="bf16", gates="post", bias=False)
    c.update(kw)
    return c


def listed() -> List[dict]:
    return [
        # the smallest call: fp32 throughout, two heads of 64, seven nodes; launches and host work only
        dict(_gdn("step", 1, 7, 1, "random", 3, Hk=2, Hv=2, d=64, dtype="f32"), name="step f32 d64 b1 n7"),
        # one request, one layer, a short MTP spine with suffix branches
        dict(_gdn("step", 1, 16, 1, "spine", 4), name="step b1 n16"),
        # one GDN layer of a serving batch: the batch the commit bar is quoted on
        dict(_gdn("step", 8, 64, 1, "random", 8), name="step b8 n64"),
        # the recurrent half of a whole hybrid model in one cycle
        dict(_gdn("step", 4, 32, 48, "random", 6), name="step 48L b4 n32"),
        # large trees, large batch
        dict(_gdn("step", 32, 256, 1, "random", 12), name="step b32 n256"),
        # one request through all 48 layers: 28 active rows padded to 32, permuted, raw gates, commit folded in
        dict(_gdn("fused", 1, 28, 48, "spine", _SPINE, rows=32, gates="raw"), name="fused 48L b1 n28"),
        # node states exported for a later cycle instead of being recomputed
        dict(_gdn("cached", 4, 32, 8, "random", 6), name="cached 8L b4 n32"),
        # one short chat request's attention layer
        dict(kind="attn", B=1, N=16, rows=16, Hq=32, Hkv=8, ctx=4000, shape="spine", depth=4, name="attn b1 ctx4k"),
        # a batch of coding-agent requests of uneven length
        dict(kind="attn", B=8, N=28, rows=32, Hq=32, Hkv=8, ctx=16384, shape="spine", depth=_SPINE, name="attn b8 ctx16k"),
        # greedy decoding of one request: argmax rows along the walk
        dict(kind="accept", mode="greedy", B=1, N=28, rows=32, V=151936, shape="spine", depth=_SPINE, name="accept greedy b1"),
        # sampled decoding of a batch: rejection sampling with residuals
        dict(kind="accept", mode="rejection", B=8, N=64, rows=64, V=151936, shape="random", depth=8, name="accept rejection b8"),
        # draft positions of a batch: five drafting steps of eight sequences
        dict(kind="select", R=40, V=151936, dtype="bf16", name="select bf16 r40"),
    ]


def _log_int(rng: random.Random, lo: int, hi: int) -> int:
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def _tree_of(rng: random.Random, N: int):
    shape = rng.choice(["random", "random", "spine", "spine", "chains", "star"])
    if shape == "random":
        depth = rng.randint(4, 12)
        while sum(2 ** k for k in range(1, depth + 1)) < N:
            depth += 1
        return shape, depth
    return shape, {"spine": rng.randint(4, _SPINE), "chains": _CHAIN, "star": 2}[shape]


def draw(rng: random.Random) -> dict:
    kind = rng.choice(["step", "step", "step", "step f32", "fused", "fused", "cached", "attn", "attn", "accept", "accept", "select"])
    if kind in ("step", "fused"):
        # up to 8192 node rows and 192 states in one call
        B, L = _log_int(rng, 1, 32), _log_int(rng, 1, 48)
        while B * L > 192:
            B, L = _log_int(rng, 1, 32), _log_int(rng, 1, 48)
        top = min(64 if kind == "fused" else 256, 8192 // (B * L))
        N = _log_int(rng, min(4, top), top)
        shape, depth = _tree_of(rng, N)
        Hk = rng.choice([16, 16, 8])
        return _gdn(kind, B, N, L, shape, depth, Hk=Hk, Hv=2 * Hk, rows=N + (-N % 32 if rng.random() < 0.5 else 0),
                    gates=rng.choice(["post", "raw"]), bias=rng.random() < 0.3)
    if kind == "step f32":
        N = _log_int(rng, 4, 64)
        shape, depth = _tree_of(rng, N)
        Hk = rng.choice([2, 4, 8])
        return _gdn("step", _log_int(rng, 1, 8), N, 1, shape, depth, Hk=Hk, Hv=Hk * rng.choice([1, 2]), d=rng.choice([64, 128]), dtype="f32")
    if kind == "cached":
        B, L = _log_int(rng, 1, 8), _log_int(rng, 1, 8)
        N = _log_int(rng, 4, min(64, 1024 // (B * L)))
        shape, depth = _tree_of(rng, N)
        return _gdn(kind, B, N, L, shape, depth)
    if kind == "attn":
        B = _log_int(rng, 1, 8)
        N = _log_int(rng, 4, 64)
        shape, depth = _tree_of(rng, N)
        return dict(kind="attn", B=B, N=N, rows=N + (-N % 32 if rng.random() < 0.5 else 0), Hq=rng.choice([32, 32, 16]), Hkv=rng.choice([8, 8, 4]),
                    ctx=_log_int(rng, 256, 131072 // B), shape=shape, depth=depth)
    if kind == "accept":
        B, V = _log_int(rng, 1, 16), _log_int(rng, 8000, 151936)
        N = _log_int(rng, 4, min(64, 8 * 64 * 151936 // (B * V)))
        shape, depth = _tree_of(rng, N)
        return dict(kind="accept", mode=rng.choice(["greedy", "rejection"]), B=B, N=N, rows=N + (-N % 32 if rng.random() < 0.5 else 0), V=V,
                    shape=shape, depth=depth)
    return dict(kind="select", R=_log_int(rng, 1, 1024), V=_log_int(rng, 8000, 151936), dtype=rng.choice(["bf16", "f32"]))


# ---------------------------------------------------------------------------
# trees and paths
# ---------------------------------------------------------------------------
def _tree(rng: random.Random, shape: str, N: int, depth: int) -> List[int]:
    """parent[i] in {-1} U [0, i); -1 is the state before the tree."""
    if shape == "star":
        return [-1] + [0] * (N - 1)
    if shape == "chains":
        return [-1 if i % _CHAIN == 0 else i - 1 for i in range(N)]
    if shape == "spine":   # a principal chain; two siblings per level, earliest levels first; the rest lengthens those branches
        s = max(1, min(depth, N // 2))
        parent = [i - 1 for i in range(s)]
        tails = []
        for lvl in range(s):
            for _ in range(2):
                if len(parent) < N:
                    parent.append(lvl - 1)
                    tails.append((len(parent) - 1, lvl + 1))
        j = 0
        while len(parent) < N:
            node, dep = tails[j % len(tails)]
            parent.append(node if dep < depth + 3 else rng.randrange(-1, s))
            tails[j % len(tails)] = (len(parent) - 1, dep + 1) if dep < depth + 3 else (parent[-1], dep)
            j += 1
        return parent
    while True:            # frontier expansion, fan-out U{1..4}
        parent, dep, frontier = [], [], [-1]
        while len(parent) < N and frontier:
            p = frontier.pop(rng.randrange(len(frontier)))
            d = 0 if p < 0 else dep[p]
            if d >= depth:
                continue
            for _ in range(rng.randint(1, 4)):
                if len(parent) < N:
                    parent.append(p)
                    dep.append(d + 1)
                    frontier.append(len(parent) - 1)
        if len(parent) == N:
            return parent


def _depths(parent: List[int]) -> List[int]:
    d: List[int] = []
    for p in parent:
        d.append(1 if p < 0 else d[p] + 1)
    return d


def _accepted(rng: random.Random, parent: List[int]) -> List[int]:
    """A walk from the root along uniformly drawn children, of geometric length."""
    kids: Dict[int, List[int]] = {}
    for i, p in enumerate(parent):
        kids.setdefault(p, []).append(i)
    n = 1
    while rng.random() >= _P_STOP:
        n += 1
    path, cur = [], -1
    while len(path) < n and kids.get(cur):
        cur = rng.choice(kids[cur])
        path.append(cur)
    return path


def _plan(case: dict, seed: int):
    """Trees, slot maps and accepted paths of one batch, on the host."""
    rng = random.Random(seed * 7919 + 17)
    B, N, rows = case["B"], case["N"], case["rows"]
    parents = [_tree(rng, case["shape"], N, case["depth"]) for _ in range(B)]
    slot = np.array([rng.sample(range(rows), N) if rows > N else list(range(N)) for _ in range(B)], dtype=np.int32)
    paths = [_accepted(rng, p) for p in parents]
    lmax = max(max(_depths(p)) for p in parents)
    acc = np.full((B, lmax), -1, dtype=np.int32)
    for b, p in enumerate(paths):
        acc[b, :len(p)] = p
    pool = list(range(B + 1))
    rng.shuffle(pool)
    return dict(parents=parents, parent=np.array(parents, dtype=np.int32), slot=slot, paths=paths, lmax=lmax,
                accepted=torch.from_numpy(acc).cuda(), length=torch.tensor([len(p) for p in paths], dtype=torch.int32, device="cuda"),
                row=torch.tensor(pool[:B], dtype=torch.int32, device="cuda"))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
class _Draws:
    """Seeded tensors drawn on the device."""

    def __init__(self, seed: int):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)

    def normal(self, *shape, dt=torch.float32, std=1.0):
        t = torch.empty(shape, dtype=torch.float32 if dt == torch.float32 else dt, device="cuda")
        return t.normal_(0.0, std, generator=self.g)

    def uniform(self, *shape, lo=0.0, hi=1.0):
        return torch.empty(shape, dtype=torch.float32, device="cuda").uniform_(lo, hi, generator=self.g)


def _gdn_cycle(r: _Draws, case: dict, p: dict, shared: dict):
    """One cycle's operand buffers of all layers and their argument blocks."""
    L, B, Ns, Hk, Hv, d, dt = case["L"], case["B"], case["rows"], case["Hk"], case["Hv"], case["d"], _DT[case["dtype"]]
    C = 2 * Hk * d + Hv * d
    t = dict(x=r.normal(L, B, Ns, C, dt=dt), q=torch.empty(L, B, Ns, Hk, d, dtype=dt, device="cuda"),
             k=torch.empty(L, B, Ns, Hk, d, dtype=dt, device="cuda"), v=torch.empty(L, B, Ns, Hv, d, dtype=dt, device="cuda"),
             out=torch.empty(L, B, Ns, Hv, d, dtype=dt, device="cuda"), status=torch.full((L, B), -1, dtype=torch.int32, device="cuda"))
    if case["gates"] == "raw":
        t["alpha"], t["beta"] = r.normal(L, B, Ns, Hv, dt=dt), r.normal(L, B, Ns, Hv, dt=dt)
    else:
        t["alpha"] = r.uniform(L, B, Ns, Hv, lo=0.9, hi=1.0).to(dt)
        t["beta"] = torch.sigmoid(r.normal(L, B, Ns, Hv)).to(dt)
    if case["kind"] == "cached":
        t["snap_out"] = torch.zeros(L, B, case["N"], Hv, d, d, device="cuda")
    layers = []
    for i in range(L):
        own = {n: v[i] for n, v in t.items()}
        own.update({n: v[i] for n, v in shared.items()})
        layers.append(binding.GdnLayer(Hk=Hk, Hv=Hv, d=d, state_row=p["row"], scale=d ** -0.5, qk_l2norm=True,
                                       snapshot_mode=2 if case["kind"] == "cached" else 0, **own))
    return t, layers, binding.Context.pack(layers)


def _prepare_gdn(case: dict, seed: int) -> dict:
    p, r = _plan(case, seed), _Draws(seed)
    L, B, Hk, Hv, d, dt = case["L"], case["B"], case["Hk"], case["Hv"], case["d"], _DT[case["dtype"]]
    C = 2 * Hk * d + Hv * d
    shared = dict(conv_w=r.normal(L, C, 4, dt=dt, std=0.5), conv_hist=r.normal(L, B + 1, 3, C, dt=dt),
                  state=r.normal(L, B + 1, Hv, d, d, std=0.02))
    if case["bias"]:
        shared["conv_b"] = r.normal(L, C, dt=dt, std=0.1)
    if case["gates"] == "raw":
        shared["a_log"] = torch.log(r.uniform(L, Hv, lo=0.02, hi=0.2))
        shared["dt_bias"] = r.uniform(L, Hv, lo=-1.0, hi=1.0)
    s = dict(p=p, shared=shared, desc=_ctx().tree_desc(p["parent"], slot=p["slot"], n_slots=case["rows"]))
    s["cycles"] = [_gdn_cycle(r, case, p, shared) for _ in range(2 if case["kind"] == "fused" else 1)]
    if case["kind"] == "fused":    # the cycle before the first timed one
        _ctx().verify(s["desc"], s["cycles"][1][2])
        s["turn"] = 0
    return s


def _prepare_attn(case: dict, seed: int) -> dict:
    p, r = _plan(case, seed), _Draws(seed)
    B, N, Ns, Hq, Hkv, bf = case["B"], case["N"], case["rows"], case["Hq"], case["Hkv"], torch.bfloat16
    rng = random.Random(seed * 31 + 5)
    ctx = [case["ctx"] if b == 0 else rng.randint((case["ctx"] + 1) // 2, case["ctx"]) for b in range(B)]   # uneven requests
    S = case["ctx"] + Ns
    t = dict(k_cache=r.normal(B + 1, S, Hkv, 128, dt=bf), v_cache=r.normal(B + 1, S, Hkv, 128, dt=bf), q=r.normal(B, N, Hq, 128, dt=bf),
             k_new=r.normal(B, N, Hkv, 128, dt=bf), v_new=r.normal(B, N, Hkv, 128, dt=bf),
             ctx_len=torch.tensor(ctx, dtype=torch.int32, device="cuda"), cache_row=p["row"],
             out=torch.empty(B, N, Hq, 128, device="cuda"), lse=torch.empty(B, N, Hq, device="cuda"),
             status=torch.full((B,), -1, dtype=torch.int32, device="cuda"))
    layer = binding.AttnLayer(Hq=Hq, Hkv=Hkv, scale=128 ** -0.5, **t)
    return dict(p=p, t=t, layer=layer, packed=binding.Context.pack_attn([layer]), ctx_len_out=torch.zeros_like(t["ctx_len"]),
                desc=_ctx().tree_desc(p["parent"], slot=p["slot"], n_slots=Ns))


def _prepare_accept(case: dict, seed: int) -> dict:
    """Target rows are peaked softmax rows; a child's proposal row is its parent's target row mixed with a row of its own,
    and its token is drawn from it.  Greedy: the target's favourite is the next node of a path of geometric length."""
    p, r = _plan(case, seed), _Draws(seed)
    B, N, Ns, V = case["B"], case["N"], case["rows"], case["V"]
    target = torch.softmax(r.normal(B, Ns + 1, V, std=3.0), dim=-1)
    token = torch.randint(0, V, (B, Ns), dtype=torch.int32, device="cuda", generator=r.g)
    s = dict(p=p, mode=case["mode"], desc=_ctx().tree_desc(p["parent"], slot=p["slot"], n_slots=Ns))
    extra = {}
    if case["mode"] == "greedy":
        for b, path in enumerate(p["paths"]):
            rows = [Ns] + [int(p["slot"][b, i]) for i in path]
            for row, child in zip(rows, path):
                target[b, row, token[b, int(p["slot"][b, child])].long()] = 0.5
    else:
        slot = torch.from_numpy(p["slot"]).long().cuda()
        par = torch.from_numpy(p["parent"]).long().cuda()
        prow = torch.where(par < 0, torch.full_like(par, Ns), torch.gather(slot, 1, par.clamp(min=0)))
        q = torch.softmax(r.normal(B, Ns, V, std=3.0), dim=-1)
        for b in range(B):
            q[b, slot[b]] = 0.6 * target[b, prow[b]] + 0.4 * q[b, slot[b]]
            token[b] = (q[b] / torch.empty_like(q[b]).exponential_(generator=r.g)).argmax(dim=-1).to(torch.int32)
        noise = torch.empty(B, V, device="cuda").exponential_(generator=r.g) + 1e-6
        extra = dict(q_draft=q, uniforms=r.uniform(B, Ns), noise=noise, work=torch.empty(B, V, device="cuda"))
    one = lambda *sh: torch.full(sh, -1, dtype=torch.int32, device="cuda")
    s["out"] = dict(accepted=one(B, p["lmax"]), length=one(B), next_token=one(B), final_node=one(B))
    s["args"] = dict(token=token, p_target=target, **extra)
    return s


def _prepare_select(case: dict, seed: int) -> dict:
    """Logits rows of three kinds in turn: plain, coarsely quantised (ties), and 70% masked with -inf."""
    r = _Draws(seed)
    R, V = case["R"], case["V"]
    x = r.normal(R, V, std=3.0)
    x[1::3] = torch.round(x[1::3])
    x[2::3].masked_fill_(torch.rand(x[2::3].shape, device="cuda", generator=r.g) < 0.7, -math.inf)
    return dict(logits=x.to(_DT[case["dtype"]]), spine=torch.zeros(R, dtype=torch.int32, device="cuda"),
                cand=torch.zeros(R, 3, dtype=torch.int32, device="cuda"))


def prepare(case: dict, seed: int) -> dict:
    make = {"step": _prepare_gdn, "fused": _prepare_gdn, "cached": _prepare_gdn, "attn": _prepare_attn, "accept": _prepare_accept,
            "select": _prepare_select}[case["kind"]]
    return dict(make(case, seed), kind=case["kind"])


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s: dict) -> dict:
    c, kind = _ctx(), s["kind"]
    if kind in ("step", "cached"):
        p, (t, _, packed) = s["p"], s["cycles"][0]
        c.verify(s["desc"], packed)
        if kind == "cached":
            return {n: t[n] for n in ("q", "k", "v", "out", "status", "snap_out")}
        c.commit(s["desc"], packed, p["accepted"], p["length"])
        return dict({n: t[n] for n in ("q", "k", "v", "out", "status")}, state=s["shared"]["state"], conv_hist=s["shared"]["conv_hist"])
    if kind == "fused":            # the two operand sets take turns, as the cycles of a request do
        p, turn = s["p"], s["turn"]
        s["turn"] = 1 - turn
        t, prev = s["cycles"][turn], s["cycles"][1 - turn]
        c.commit_verify(s["desc"], prev[2], p["accepted"], p["length"], s["desc"], t[2])
        return dict({n: t[0][n] for n in ("q", "k", "v", "out", "status")}, state=s["shared"]["state"], conv_hist=s["shared"]["conv_hist"])
    if kind == "attn":
        p, t = s["p"], s["t"]
        c.kv_write_tree(s["desc"], s["packed"])
        c.tree_attention(s["desc"], s["packed"])
        c.kv_publish(s["desc"], s["packed"], p["accepted"], p["length"], s["ctx_len_out"])
        return dict({n: t[n] for n in ("out", "lse", "status", "k_cache", "v_cache")}, ctx_len=s["ctx_len_out"])
    if kind == "accept":
        c.accept(s["desc"], mode=s["mode"], **s["args"], **s["out"])
        return s["out"]
    c.select_spine_top3(s["logits"], s["spine"], s["cand"])
    return {"spine": s["spine"], "cand": s["cand"]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case: dict) -> dict:
    kind = case["kind"]
    if kind in ("step", "fused", "cached"):
        B, N, L, Hk, Hv, d = (case[n] for n in ("B", "N", "L", "Hk", "Hv", "d"))
        C, e = 2 * Hk * d + Hv * d, 4 if case["dtype"] == "f32" else 2
        state = 4 * B * Hv * d * d
        # in: state, x, gates, taps and (read once each) history; out: recorded operands, outputs, states
        n_bytes = state + B * N * C * e + 2 * B * N * Hv * e + 4 * C * e + 3 * B * C * e + B * N * C * e + B * N * Hv * d * e
        n_bytes += N * state if kind == "cached" else state + 3 * B * C * e
        return {"bytes": float(L * n_bytes), "flops": float(L * (B * N * Hv * 7 * d * d + 12 * B * N * C))}
    if kind == "attn":
        B, N, Hq, Hkv = (case[n] for n in ("B", "N", "Hq", "Hkv"))
        keys = case["ctx"] * (1 + 0.75 * (B - 1)) + B * N      # half to full length, one sequence at full length
        return {"bytes": float(keys * Hkv * 512 + B * N * Hkv * 512 + B * N * Hq * (2 * 128 + 4 * 128 + 4)),
                "flops": float(4 * 128 * keys * N * Hq)}
    if kind == "accept":
        # rows of a walk of mean geometric length: one target row per accepted node and one at its end; with rejection sampling
        # one proposal row per refused child, and the race's variates
        rows = 1 / _P_STOP + 1 if case["mode"] == "greedy" else 8
        return {"bytes": float(4 * case["B"] * case["V"] * rows), "flops": 0.0}
    return {"bytes": float(case["R"] * case["V"] * (2 if case["dtype"] == "bf16" else 4) + 16 * case["R"]), "flops": 0.0}


def tolerance(case: dict):
    """bf16 results and operands: one rounding in the last of eight bits.  fp32 results of fp32 inputs: summation order.  Attention:
    probabilities enter the second product as bf16.  Token and node numbers are unique."""
    if case["kind"] in ("accept", "select"):
        return "exact"
    return {"rel": 1e-5} if case.get("dtype") == "f32" else {"rel": 5e-3}
