"""The work that a user of this package has it do, as measurable cases.

A Mamba drafter uses the library in four ways: it encodes a context (one call per layer, or a whole stack of layers), drafts
a tree below it (one round = every level of every layer, replayed from a CUDA graph at batch 1, launched at batch > 1),
runs its block stack for one generation of that tree (projections included), and, for a Mamba-2 drafter, does the first two
with SSD layers.  The shapes are the repository's five configurations (a 130M drafter: 24 layers, 1536 channels; contexts
of 256 to 32768 tokens; trees of 15 to 150 nodes; a batch of 32 sequences) plus ragged ones; values follow the input recipe
of those configurations (x, z, B, C ~ N(0, 1); step sizes inside [1e-3, 1e-1]; A = -(1..16), or that perturbed as training
would leave it).
"""

from __future__ import annotations

import math
import random

import torch

import paper_2506_01206_b200 as md
from paper_2506_01206_b200.drafter import ToyDrafter
from paper_2506_01206_b200.stack import DrafterStack, RoundGraphCache

N, W = 16, 4            # states and conv taps of an S6 layer
HEAD, SSD_N = 64, 128   # channels per head and states of an SSD layer
DT_BIAS = -4.579712     # softplus(bias + 0.5 N(0, 1)) stays inside [1e-3, 1e-1]
DT_CLIP = 2.3125
VOCAB, D_MODEL, DT_RANK = 50280, 768, 48
LARGEST = 24 * 32768 * 1536   # layers x tokens x channels of the largest listed encode


def listed():
    return [
        # The smallest use: the fp32 configuration, encode 256 tokens, draft a 15-node tree, commit (launches and latency).
        {"name": "tiny step fp32", "kind": "step", "layers": 1, "d_inner": 64, "act": "f32", "n_seq": 1, "lo": 256, "hi": 256,
         "lens_seed": 0, "general_A": False, "init": False, "branching": "2,2,2", "cap": 0},
        # Context encode of the whole 130M stack, the benchmark's own context length.
        {"name": "stack encode 2k", "kind": "stack_encode", "layers": 24, "d_inner": 1536, "act": "bf16", "n_seq": 1, "lo": 2048,
         "hi": 2048, "lens_seed": 0, "general_A": False, "init": False},
        # The long-context configuration.
        {"name": "stack encode 32k", "kind": "stack_encode", "layers": 24, "d_inner": 1536, "act": "bf16", "n_seq": 1, "lo": 32768,
         "hi": 32768, "lens_seed": 0, "general_A": False, "init": False},
        # One layer of the batched configuration: 32 packed sequences of 1k to 8k tokens.
        {"name": "layer encode packed 32", "kind": "layer_encode", "layers": 1, "d_inner": 1536, "act": "bf16", "n_seq": 32, "lo": 1024,
         "hi": 8192, "lens_seed": 0, "general_A": False, "init": False},
        # One layer of a trained drafter (A no longer the initial pattern), the next piece of a context: odd length, from a slot.
        {"name": "layer encode trained A", "kind": "layer_encode", "layers": 1, "d_inner": 1536, "act": "bf16", "n_seq": 1, "lo": 1777,
         "hi": 1777, "lens_seed": 0, "general_A": True, "init": True},
        # fp32 activations, three ragged sequences, a width that fills no whole block.
        {"name": "layer encode fp32 ragged", "kind": "layer_encode", "layers": 1, "d_inner": 1000, "act": "f32", "n_seq": 3, "lo": 300,
         "hi": 1500, "lens_seed": 1, "general_A": True, "init": False},
        # The draft round of the 150-node configuration, all 24 layers and the commit, as a drafter replays it.
        {"name": "draft round 150", "kind": "round", "layers": 24, "d_inner": 1536, "act": "bf16", "branching": "4,4,2,2,2", "cap": 150},
        # The batched configuration's round: 32 sequences with a random 32-node tree each.
        {"name": "draft round 32 x 32", "kind": "batch_round", "layers": 24, "d_inner": 1536, "act": "bf16", "n_seq": 32, "nodes": 32,
         "levels": 5, "tree_seed": 0},
        # One generation of the block stack: the widest level of the paper's (3,3,2,1) tree, projections inside the step ...
        {"name": "generation 18", "kind": "generation", "width": 18, "fused": True},
        # ... and the drafter's default mode on a single chain.
        {"name": "generation 1 split", "kind": "generation", "width": 1, "fused": False},
        # A Mamba-2 layer: context encode and the 150-node round.
        {"name": "ssd encode 2k", "kind": "ssd_encode", "d_inner": 1536, "n_seq": 1, "lo": 2048, "hi": 2048, "lens_seed": 0, "init": False},
        {"name": "ssd round 150", "kind": "ssd_round", "d_inner": 1536, "branching": "4,4,2,2,2", "cap": 150},
    ]


# ---------------------------------------------------------------- more cases of the same ranges
def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _width(rng):
    return 8 * _log(rng, 8, 256)


def _branching(rng):
    """Branching factors of a tree of at most 150 nodes."""
    while True:
        b = [rng.randint(1, 4) for _ in range(rng.randint(1, 6))]
        n, w = 1, 1
        for f in b:
            w *= f
            n += w
        if n <= 150:
            return ",".join(str(f) for f in b)


def draw(rng):
    kind = rng.choice(["step", "stack_encode", "layer_encode", "round", "batch_round", "generation", "ssd_encode", "ssd_round"])
    if kind == "generation":
        return {"kind": kind, "width": _log(rng, 1, 64), "fused": rng.random() < 0.5}
    if kind == "ssd_round":
        return {"kind": kind, "d_inner": HEAD * _log(rng, 1, 32), "branching": _branching(rng), "cap": 0}
    if kind == "ssd_encode":
        n_seq, hi = _log(rng, 1, 8), _log(rng, 16, 8192)
        return {"kind": kind, "d_inner": HEAD * _log(rng, 1, 32), "n_seq": n_seq, "lo": max(1, hi // rng.randint(1, 4)), "hi": hi,
                "lens_seed": rng.randrange(1000), "init": rng.random() < 0.3}
    act = rng.choice(["bf16", "bf16", "f32"])
    if kind == "round":
        return {"kind": kind, "layers": _log(rng, 1, 24), "d_inner": _width(rng), "act": act, "branching": _branching(rng), "cap": 0}
    if kind == "batch_round":
        return {"kind": kind, "layers": _log(rng, 1, 24), "d_inner": min(_width(rng), 1536), "act": act, "n_seq": _log(rng, 2, 48),
                "nodes": rng.randint(8, 40), "levels": 5, "tree_seed": rng.randrange(1000)}
    c = {"kind": kind, "layers": 1, "d_inner": _width(rng), "act": act}
    if kind == "step":
        c.update(layers=_log(rng, 1, 8), d_inner=min(c["d_inner"], 768), n_seq=1, hi=_log(rng, 32, 1024))
    elif kind == "stack_encode":
        c.update(layers=_log(rng, 2, 24), n_seq=_log(rng, 1, 8), hi=_log(rng, 64, 16384))
    else:
        c.update(n_seq=_log(rng, 1, 32), hi=_log(rng, 64, 16384))
    while c["layers"] * c["n_seq"] * c["hi"] * c["d_inner"] * (2 if act == "f32" else 1) > LARGEST // 2:
        c["hi"] = c["hi"] * 2 // 3
    c["lo"] = max(1, c["hi"] // rng.randint(1, 4))
    c.update(lens_seed=rng.randrange(1000), general_A=rng.random() < 0.5, init=rng.random() < 0.3)
    if kind == "step":
        c.update(branching=_branching(rng), cap=0)
    return c


# ---------------------------------------------------------------- what a case's sizes mean
def _lens(c):
    r = random.Random(c["lens_seed"])
    return [r.randint(c["lo"], c["hi"]) for _ in range(c["n_seq"])]


def _tree(c):
    """(parents, level offsets) of the case's tree in breadth-first order; the deepest level is cut to `cap` nodes in all."""
    levels, first = [[-1]], 0
    for f in (int(v) for v in c["branching"].split(",")):
        prev = levels[-1]
        levels.append([first + j for j in range(len(prev)) for _ in range(f)])
        first += len(prev)
    total = sum(len(v) for v in levels)
    if c["cap"] and total > c["cap"]:
        keep = len(levels[-1]) - (total - c["cap"])
        levels[-1] = sorted(random.Random(0).sample(levels[-1], keep))
    return _flat(levels)


def _random_tree(nodes, depth, rng):
    """A tree of exactly `nodes` nodes on at most `depth` levels, 1 to 3 children a node, as lists of parents per level."""
    levels, total = [[-1]], 1
    first = 0
    for l in range(depth - 1):
        prev = levels[-1]
        nxt = [first + j for j in range(len(prev)) for _ in range(rng.randint(1, 3))]
        first += len(prev)
        left = nodes - total
        if l == depth - 2 and len(nxt) < left:   # the last level takes what is missing
            nxt = sorted(nxt + [first - len(prev) + rng.randrange(len(prev)) for _ in range(left - len(nxt))])
        nxt = nxt[:left]
        if not nxt:
            break
        levels.append(nxt)
        total += len(nxt)
    return levels


def _flat(levels):
    off = [0]
    for v in levels:
        off.append(off[-1] + len(v))
    return [p for v in levels for p in v], off


def _batch_trees(c):
    """All sequences' trees merged level by level: (sequence, parent's index or -1) per node, and the level offsets."""
    rng = random.Random(c["tree_seed"])
    trees = [_random_tree(c["nodes"], c["levels"], rng) for _ in range(c["n_seq"])]
    nodes, off, index = [], [0], {}
    for l in range(c["levels"]):
        for s, t in enumerate(trees):
            if l >= len(t):
                continue
            base = sum(len(v) for v in t[:l])
            for j, p in enumerate(t[l]):
                index[s, base + j] = len(nodes)
                nodes.append((s, -1 if p < 0 else index[s, p]))
        off.append(len(nodes))
    return nodes, off


# ---------------------------------------------------------------- inputs
def _act(c):
    return {"f32": torch.float32, "bf16": torch.bfloat16}[c.get("act", "bf16")]


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _normal(g, shape, dtype, scale=1.0):
    t = torch.empty(shape, dtype=dtype, device="cuda").normal_(generator=g)
    return t if scale == 1.0 else t.mul_(scale)


def _activations(g, layers, rows, d, dt_cols, n, act, bc_scale=1.0):
    """Stacked (layers, rows, .) tensors x, z, dt, B, C."""
    x, z = _normal(g, (layers, rows, d), act), _normal(g, (layers, rows, d), act)
    dt = _normal(g, (layers, rows, dt_cols), act, 0.5).clamp_(-DT_CLIP, DT_CLIP)
    return x, z, dt, _normal(g, (layers, rows, n), act, bc_scale), _normal(g, (layers, rows, n), act, bc_scale)


def _layers(g, c):
    d, out = c["d_inner"], []
    for _ in range(c["layers"]):
        A = -torch.arange(1, N + 1, dtype=torch.float32, device="cuda").repeat(d, 1)
        flags = md.MDRAFT_DT_SOFTPLUS
        if c.get("general_A"):
            A = A * torch.exp(0.25 * _normal(g, (d, N), torch.float32))
        else:
            flags |= md.MDRAFT_A_POWERS
        out.append(md.Layer(A.contiguous(), torch.ones(d, device="cuda"), _normal(g, (d, W), torch.float32, 0.5), None,
                            torch.full((d,), DT_BIAS, device="cuda"), _act(c), flags))
    return out


def _ssd_layer(g, c):
    d = c["d_inner"]
    h = d // HEAD
    A = -(1.0 + 15.0 * torch.arange(h, dtype=torch.float32, device="cuda") / max(h - 1, 1))
    return md.SsdLayer(A.contiguous(), torch.ones(d, device="cuda"), _normal(g, (d, W), torch.float32, 0.5), None,
                       torch.full((h,), DT_BIAS, device="cuda"))


def _i32(v):
    return torch.tensor(v, dtype=torch.int32, device="cuda")


def _fill_slots(g, cache, slots):
    """States as an encode leaves them: of order one, in every layer of the named slots."""
    cache.ssm[:, slots] = _normal(g, cache.ssm[:, slots].shape, torch.float32)
    cache.conv[:, slots] = _normal(g, cache.conv[:, slots].shape, cache.conv.dtype)


def _rows(stacked):
    return [tuple(t[l] for t in stacked) for l in range(stacked[0].shape[0])]


def _offsets(c):
    """(cu_seqlens or None for one sequence, total tokens, longest, final slots, starting slots or None)."""
    lens = _lens(c)
    cu = [0]
    for n in lens:
        cu.append(cu[-1] + n)
    s = len(lens)
    return (_i32(cu) if s > 1 else None, cu[-1], max(lens), _i32(list(range(s))), _i32(list(range(s, 2 * s))) if c["init"] else None)


def prepare(case, seed):
    return {"step": _prepare_step, "stack_encode": _prepare_encode, "layer_encode": _prepare_encode, "round": _prepare_round,
            "batch_round": _prepare_batch_round, "generation": _prepare_generation, "ssd_encode": _prepare_ssd_encode,
            "ssd_round": _prepare_ssd_round}[case["kind"]](case, _gen(seed))


def _prepare_encode(c, g, extra_slots=0):
    cu, T, longest, final, init = _offsets(c)
    layers = _layers(g, c)
    stacked = _activations(g, c["layers"], T, c["d_inner"], c["d_inner"], N, _act(c))
    out = torch.zeros((c["layers"], T, c["d_inner"]), dtype=_act(c), device="cuda")
    stack = DrafterStack(layers, 2 * c["n_seq"] + extra_slots, T, c["n_seq"], longest)
    if init is not None:
        _fill_slots(g, stack.cache, list(range(c["n_seq"], 2 * c["n_seq"])))
    return {"kind": c["kind"], "stack": stack, "inputs": _rows(stacked), "out": out, "outs": list(out), "cu": cu, "longest": longest,
            "final": final, "init": init}


def _prepare_step(c, g):
    parents, off = _tree(c)
    m, s = len(parents), 2 * c["n_seq"]
    st = _prepare_encode(c, g, extra_slots=m)
    nodes = _activations(g, c["layers"], m, c["d_inner"], c["d_inner"], N, _act(c))
    node_out = torch.zeros((c["layers"], m, c["d_inner"]), dtype=_act(c), device="cuda")
    st.update(nodes=_rows(nodes), node_out=node_out, node_outs=list(node_out), offsets=off,
              parent=_i32([0 if p < 0 else s + p for p in parents]), node=_i32([s + i for i in range(m)]), accepted=_i32([s + m - 1]))
    return st


def _prepare_round(c, g):
    parents, off = _tree(c)
    m = len(parents)
    stack = DrafterStack(_layers(g, c), 1 + m, 1, 1, 1)
    rounds = RoundGraphCache(stack, m)
    rounds.node_slot.copy_(_i32([1 + i for i in range(m)]))
    rounds.parent_slot.copy_(_i32([0 if p < 0 else 1 + p for p in parents]))
    rounds.accepted_slot.fill_(m)
    rounds.run(off)   # a drafter meets a tree shape once and replays it from then on
    for mine, t in zip((rounds.x, rounds.z, rounds.dt, rounds.B, rounds.C),
                       _activations(g, c["layers"], m, c["d_inner"], c["d_inner"], N, _act(c))):
        for l in range(c["layers"]):
            mine[l].copy_(t[l])
    _fill_slots(g, stack.cache, [0])
    return {"kind": c["kind"], "rounds": rounds, "offsets": off}


def _prepare_batch_round(c, g):
    nodes, off = _batch_trees(c)
    m, s = len(nodes), c["n_seq"]
    stack = DrafterStack(_layers(g, c), s + m, 1, 1, 1)
    stacked = _activations(g, c["layers"], m, c["d_inner"], c["d_inner"], N, _act(c))
    out = torch.zeros((c["layers"], m, c["d_inner"]), dtype=_act(c), device="cuda")
    _fill_slots(g, stack.cache, list(range(s)))
    last = [max(i for i, (q, _) in enumerate(nodes) if q == k) for k in range(s)]
    return {"kind": c["kind"], "stack": stack, "nodes": _rows(stacked), "node_out": out, "node_outs": list(out), "offsets": off,
            "parent": _i32([q if p < 0 else s + p for q, p in nodes]), "node": _i32([s + i for i in range(m)]),
            "accepted": _i32([s + i for i in last]), "sequence": _i32(list(range(s)))}


def _prepare_generation(c, g):
    w = c["width"]
    up = (w + 1) // 2   # the level above: two children a node
    d = ToyDrafter(d_model=D_MODEL, dt_rank=DT_RANK, vocab=VOCAB, max_nodes=up + w, seed=int(g.initial_seed()), fused=c["fused"])
    d.tokens.copy_(torch.randint(0, VOCAB, (up + w,), generator=g, device="cuda"))
    d.node_slot.copy_(_i32([1 + i for i in range(up + w)]))
    d.parent_slot.copy_(_i32([0] * up + [1 + j // 2 for j in range(w)]))
    d.generation(up, up + w)   # the graph of this level, kept by the drafter
    _fill_slots(g, d.cache, list(range(1 + up)))
    return {"kind": c["kind"], "drafter": d, "lo": up, "hi": up + w}


def _prepare_ssd_encode(c, g):
    cu, T, longest, final, init = _offsets(c)
    lay, d = _ssd_layer(g, c), c["d_inner"]
    x, z, dt, B, C = (t[0] for t in _activations(g, 1, T, d, d // HEAD, SSD_N, torch.bfloat16, (N / SSD_N) ** 0.5))
    cache = md.StateCache(1, 2 * c["n_seq"], d, d_state=SSD_N)
    if init is not None:
        _fill_slots(g, cache, list(range(c["n_seq"], 2 * c["n_seq"])))
    ws = torch.empty(max(256, md.mdraft_ssd_prefill_workspace_bytes(lay, T, c["n_seq"])), dtype=torch.uint8, device="cuda")
    return {"kind": c["kind"], "layer": lay, "cache": cache, "inputs": (x, z, dt, B, C), "out": torch.zeros_like(x), "cu": cu,
            "final": final, "init": init, "ws": ws, "status": _i32([0])}


def _prepare_ssd_round(c, g):
    parents, off = _tree(c)
    m, d = len(parents), c["d_inner"]
    lay = _ssd_layer(g, c)
    ins = tuple(t[0] for t in _activations(g, 1, m, d, d // HEAD, SSD_N, torch.bfloat16, (N / SSD_N) ** 0.5))
    cache = md.StateCache(1, 1 + m, d, d_state=SSD_N)
    _fill_slots(g, cache, [0])
    return {"kind": c["kind"], "layer": lay, "cache": cache, "inputs": ins, "out": torch.zeros_like(ins[0]), "offsets": off,
            "parent": _i32([0 if p < 0 else 1 + p for p in parents]), "node": _i32([1 + i for i in range(m)]), "status": _i32([0])}


# ---------------------------------------------------------------- one pass
def run(s):
    kind = s["kind"]
    if kind == "layer_encode":
        st = s["stack"]
        md.mdraft_conv_scan_prefill(st.layers[0], st.cache, 0, *s["inputs"][0], s["outs"][0], s["cu"], s["longest"], s["init"], s["final"],
                                    st.workspace, 0, st.status)
        return s["out"], st.cache.ssm, st.cache.conv
    if kind == "stack_encode":
        st = s["stack"]
        st.prefill(s["inputs"], s["outs"], s["cu"], s["longest"], s["init"], s["final"])
        return s["out"], st.cache.ssm, st.cache.conv
    if kind == "step":
        st = s["stack"]
        st.prefill(s["inputs"], s["outs"], s["cu"], s["longest"], s["init"], s["final"])
        st.tree_round(s["nodes"], s["node_outs"], s["parent"], s["node"], s["offsets"])
        st.commit(s["accepted"], s["final"])
        return s["out"], s["node_out"], st.cache.ssm, st.cache.conv
    if kind == "round":
        r = s["rounds"]
        r.run(s["offsets"])
        return r.out, r.stack.cache.ssm, r.stack.cache.conv
    if kind == "batch_round":
        st = s["stack"]
        st.tree_round(s["nodes"], s["node_outs"], s["parent"], s["node"], s["offsets"])
        st.commit(s["accepted"], s["sequence"])
        return s["node_out"], st.cache.ssm, st.cache.conv
    if kind == "generation":
        d = s["drafter"]
        d.generation(s["lo"], s["hi"])
        return d.logits, d.cache.ssm, d.cache.conv
    if kind == "ssd_encode":
        md.mdraft_ssd_prefill(s["layer"], s["cache"], 0, *s["inputs"], s["out"], s["cu"], s["init"], s["final"], s["ws"], s["status"])
        return s["out"], s["cache"].ssm, s["cache"].conv
    md.mdraft_ssd_tree_step(s["layer"], s["cache"], 0, *s["inputs"], s["out"], s["parent"], s["node"], s["offsets"], s["status"])
    return s["out"], s["cache"].ssm, s["cache"].conv


# ---------------------------------------------------------------- what a pass cannot do without
def _slot_bytes(d, n, es):
    return d * n * 4 + (W - 1) * d * es


def _token_flops(n):
    # conv 8, two SiLU 8, softplus 6, skip and gate 4, and per state the decay 2, the update 3, the contraction with C 2
    return 26 + 7 * n


def _encode_work(c, n, dt_cols, es):
    T, d, s = sum(_lens(c)), c["d_inner"], c["n_seq"]
    return T * (3 * d + dt_cols + 2 * n) * es + (2 if c["init"] else 1) * s * _slot_bytes(d, n, es), T * d * _token_flops(n)


def _tree_work(nodes, parents, d, n, dt_cols, es):
    """Every node: its inputs read, its output, state and window written; every distinct parent read once."""
    m = nodes
    return m * (3 * d + dt_cols + 2 * n) * es + (m + parents) * _slot_bytes(d, n, es), m * d * _token_flops(n)


def work(case):
    c, kind = case, case["kind"]
    es = 4 if c.get("act") == "f32" else 2
    b = f = 0.0
    layers = c.get("layers", 1)
    if kind in ("step", "stack_encode", "layer_encode"):
        b, f = _encode_work(c, N, c["d_inner"], es)
    if kind in ("step", "round"):
        parents, _ = _tree(c)
        tb, tf = _tree_work(len(parents), len(set(parents)), c["d_inner"], N, c["d_inner"], es)
        b, f = b + tb + 2 * _slot_bytes(c["d_inner"], N, es), f + tf
    if kind == "batch_round":
        nodes, _ = _batch_trees(c)
        b, f = _tree_work(len(nodes), len({(q if p < 0 else -1, p) for q, p in nodes}), c["d_inner"], N, c["d_inner"], es)
        b += 2 * c["n_seq"] * _slot_bytes(c["d_inner"], N, es)
    if kind == "generation":
        w, d, layers = c["width"], 1536, 1
        per_layer = D_MODEL * 2 * d + d * (DT_RANK + 2 * N) + DT_RANK * d + d * D_MODEL
        tb, tf = _tree_work(w, (w + 1) // 2, d, N, 0, 2)
        b = 24 * (2 * per_layer + tb - w * 2 * (3 * d + 2 * N)) + 2 * D_MODEL * VOCAB + 2 * w * (VOCAB + D_MODEL)
        f = 24 * (2.0 * w * per_layer + tf) + 2.0 * w * D_MODEL * VOCAB
    if kind == "ssd_encode":
        b, f = _encode_work(c, SSD_N, c["d_inner"] // HEAD, 2)
    if kind == "ssd_round":
        parents, _ = _tree(c)
        b, f = _tree_work(len(parents), len(set(parents)), c["d_inner"], SSD_N, c["d_inner"] // HEAD, 2)
    return {"bytes": float(layers * b), "flops": float(layers * f)}


def tolerance(case):
    kind = case["kind"]
    if kind == "generation":
        return {"rel": 2e-2, "max": 0.2}      # 24 layers of bf16 activations and a bf16 residual stream
    if kind == "ssd_encode":
        return {"rel": 1e-2, "max": 0.1}      # bf16 operands of the chunk-local products
    if case.get("act") == "f32":
        return {"rel": 2e-5, "max": 1e-3}     # 32-bit sums in another order, approximate exponentials
    return {"rel": 3e-3, "max": 2e-2}         # the output's own rounding to bf16
