#!/usr/bin/env python
"""Benchmark of the Mamba-drafter hot path on B200: one JSON line on stdout.

A "step" is one pass of the whole path over one batch of synthetic input shaped like the paper's drafter
workload (Mamba-130M: 24 layers, d_inner 1536, d_state 16; context 2048 tokens; bf16 activations, fp32 state):
  prefill of all layers (conv1d+SiLU -> Delta -> S6 scan -> gate)  ->  one draft round over a 150-node tree
  (6 levels, all layers, states forked by parent index)  ->  commit of a random accepted node.
`value` = prefill token*channels of the step / whole step time (so tree and commit time count against it);
the per-phase throughputs (prefill token*channels/s, tree node-updates/s) are reported beside it.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]
    python bench.py --profile-case prefill|stack|tree|proj|ssd|generation [sizes ...] (small runs of one kernel family for a profiler)

N > 1 (under torchrun) runs N independent replicas (the path has no exchange step): weak scaling.
`--impl reference` times the fp64 CPU oracle on a bounded sample of the same workload.
"""

from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import gen  # noqa: E402

METRIC = "s6_prefill_token_channels_per_s"
UNIT = "token*channels/s"
WORKLOAD = "cfg1 prefill (24 layers x 2048 tokens x 1536 channels, bf16/fp32-state) + cfg2 draft round (150-node tree, 6 levels) + commit"


def load_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        j = json.load(open(p))
        return float(j["hbm_gbs"]), "measured (MEASURED_PEAKS.json, copy bandwidth)"
    return 6650.0, "fallback (earlier pool measurement; MEASURED_PEAKS.json absent)"


# ----------------------------------------------------------------------------------------------- workload
class Workload:
    """cfg 2 = cfg 1's prefill followed by tree drafting; all tensors generated on the host, seeded."""

    def __init__(self, seed: int, n_layers: int = 24, general_A: bool = False):
        self.cfg = gen.get_config(2)
        c = self.cfg
        self.cfg = gen.Config(c.cid, c.name, n_layers, c.d_inner, c.d_state, c.d_conv, c.act, c.n_seq, c.context, c.tree, c.rounds, seed)
        self.n_layers = n_layers
        self.T = self.cfg.context[0]
        self.tree = gen.config_tree(self.cfg, 0)
        self.M = self.tree.n_nodes
        self.accepted = gen.random_accepted_node(self.tree, seed, self.cfg.cid, 0)
        self.params = [gen.layer_params(self.cfg, l, general_A=general_A) for l in range(n_layers)]
        self.general_A = general_A
        self._prefill = None
        self._nodes = None

    def prefill_inputs(self, l):
        return gen.prefill_inputs(self.cfg, l, self.T)

    def node_inputs(self, l):
        return gen.node_inputs(self.cfg, l, 0, self.M)

    # algorithmic bytes: activations in/out + B,C + final state write
    def prefill_bytes_per_layer(self):
        D, N, T, es = self.cfg.d_inner, self.cfg.d_state, self.T, 2
        return 4 * es * T * D + 2 * N * es * T + D * N * 4 + 3 * D * es

    def tree_bytes_per_layer(self):
        D, N, es = self.cfg.d_inner, self.cfg.d_state, 2
        state = D * N * 4 + 3 * D * es
        own = state + 3 * D * es + D * es + 2 * N * es          # child state write, x/z/dt in, out, B/C
        distinct_parents = len(set(int(p) for p in self.tree.parents))
        return self.M * own + distinct_parents * state

    def commit_bytes(self):
        D, N, es = self.cfg.d_inner, self.cfg.d_state, 2
        return 2 * (D * N * 4 + 3 * D * es) * self.n_layers


# ----------------------------------------------------------------------------------------------- clocks
class ClockSampler:
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.path = tempfile.mktemp(suffix=".csv")
        self.proc = None
        self.idx = gpu_index

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.Q}", "--format=csv,noheader,nounits", "-lms", "50",
                                          "-i", str(self.idx)], stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def stop(self):
        out = {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": 0}
        if self.proc is None:
            return out
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        sm, mx, reasons = [], [], set()
        try:
            for line in open(self.path):
                f = [v.strip() for v in line.split(",")]
                if len(f) < 9:
                    continue
                try:
                    sm.append(float(f[1])); mx.append(float(f[2]))
                except ValueError:
                    continue
                for name, v in zip(("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"), f[5:9]):
                    if v.lower().startswith("active"):
                        reasons.add(name)
            os.unlink(self.path)
        except Exception:
            pass
        if sm:
            out.update(sm_mhz=statistics.median(sm), sm_max_mhz=max(mx), samples=len(sm))
        out["reasons"] = sorted(reasons)
        return out


# ----------------------------------------------------------------------------------------------- CPU oracle leg
def time_oracle_sample(w: Workload, n_layers: int, threads: int):
    """Oracle on `n_layers` layers of the workload (prefill + the draft tree + commit by indexing)."""
    import oracle
    used = oracle.set_threads(threads)
    ins = [(w.prefill_inputs(l), w.node_inputs(l)) for l in range(n_layers)]
    lays = [oracle.layer_from_params(w.params[l]) for l in range(n_layers)]
    ins64 = [tuple(tuple(a.astype(np.float64) for a in part) for part in pair) for pair in ins]
    t0 = time.perf_counter()
    for l in range(n_layers):
        pin, nin = ins64[l]
        _, conv, h = oracle.prefill(lays[l], *pin)
        _, tconv, th = oracle.tree(lays[l], w.tree.parents, *nin, conv[0], h[0])
        _ = (tconv[w.accepted].copy(), th[w.accepted].copy())
    dt = time.perf_counter() - t0
    units = n_layers * w.T * w.cfg.d_inner
    return units / dt, dt, used


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    cores = os.cpu_count() or 1
    w = Workload(seed=0, n_layers=24)
    sample_layers = 2
    vals = []
    for _ in range(args.warmup):
        time_oracle_sample(w, 1, cores)
    t_all = 0.0
    for _ in range(args.steps):
        v, dt, used = time_oracle_sample(w, sample_layers, cores)
        vals.append(v); t_all += dt
    value = sample_layers * w.T * w.cfg.d_inner * args.steps / t_all
    sample = f"{sample_layers} of 24 layers per step (prefill 2048 tokens + 150-node tree path by path + commit), fp64, all host cores"
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": 1e3 * t_all / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": WORKLOAD, "sample": sample},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": used, "kind": "oracle", "sample": sample},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        "gpu_launches": 0,
    }
    print(json.dumps(line))


# ----------------------------------------------------------------------------------------------- GPU leg
# fp32 lane-operations per token*channel of a single-pass prefill: conv 4 + SiLU 3 + softplus 5 + step*input 1 +
# 16 states x (form the decay, decay*h, input*B, C*h) 64 + skip 1 + gate 4
ALU_LANE_OPS_PER_UNIT = 82
FP32_LANES_PER_SM, SM_COUNT, SM_MAX_MHZ = 128, 148, 1965.0
def ncu_traffic(key):
    """dram__bytes_read.sum + dram__bytes_write.sum per launch of the named kernel, from the ncu capture recorded in
    profiles/traffic.json, or None when a source file of that kernel has changed since the capture (the record keeps
    the SHA-256 of the sources it was taken with, so a stale figure cannot be reported by accident)."""
    import hashlib
    try:
        rec = json.load(open(os.path.join(ROOT, "profiles", "traffic.json")))[key]
        for rel, digest in rec["sources_sha256"].items():
            if hashlib.sha256(open(os.path.join(ROOT, rel), "rb").read()).hexdigest() != digest:
                return None, rec.get("kernel")
        return float(rec["dram_bytes_per_launch"]), rec.get("kernel")
    except Exception:
        return None, None


class BatchedTree:
    """The batched-serving draft round (32 sequences x 32-node trees): where the tree step moves tens of MB per launch."""

    def __init__(self, seed: int):
        c = gen.get_config(4)
        self.cfg = gen.Config(c.cid, c.name, c.n_layers, c.d_inner, c.d_state, c.d_conv, c.act, c.n_seq, c.context, c.tree, c.rounds, seed)
        S = self.cfg.n_seq
        trees = [gen.config_tree(self.cfg, 0, s) for s in range(S)]
        off = np.cumsum([0] + [t.n_nodes for t in trees])
        parent, nodes, lvl = [], [], [0]
        for l in range(max(t.n_levels for t in trees)):  # level-major over all sequences
            for s, t in enumerate(trees):
                if l >= t.n_levels:
                    continue
                for i in range(int(t.level_offsets[l]), int(t.level_offsets[l + 1])):
                    par = int(t.parents[i])
                    parent.append(s if par < 0 else S + int(off[s]) + par)
                    nodes.append(S + int(off[s]) + i)
            lvl.append(len(nodes))
        self.parent, self.nodes, self.levels, self.S, self.M = parent, nodes, lvl, S, len(nodes)

    def level_bytes(self, lo, hi):
        D, N, es = self.cfg.d_inner, self.cfg.d_state, 2
        state = D * N * 4 + 3 * D * es
        own = state + 3 * D * es + D * es + 2 * N * es
        return (hi - lo) * own + len(set(self.parent[lo:hi])) * state


def run_ours(args):
    import torch
    import paper_2506_01206_b200 as md
    from paper_2506_01206_b200 import replicas
    from paper_2506_01206_b200.device_inputs import i32, to_device, torch_act, upload_layer
    from paper_2506_01206_b200.stack import DrafterStack

    rank, local, world = replicas.env_ranks()
    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device; there is no CPU path")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    replicas.init("nccl", dev)
    md.load_library()

    def barrier():
        replicas.barrier(world)

    def max_over_ranks(v: float) -> float:
        return replicas.max_over_ranks(v, world, dev)

    w = Workload(seed=replicas.replica_seed(0, rank), n_layers=24)
    tdt = torch_act(w.cfg.act)
    T, M, D, NL = w.T, w.M, w.cfg.d_inner, w.n_layers

    # host copies (pinned, already in the activation dtype) and device-resident copies
    host_pre, host_node, dev_pre, dev_node = [], [], [], []
    for l in range(NL):
        hp = [to_device(a, tdt, pinned=True) for a in w.prefill_inputs(l)]
        hn = [to_device(a, tdt, pinned=True) for a in w.node_inputs(l)]
        host_pre.append(hp); host_node.append(hn)
        dev_pre.append([t.to(dev) for t in hp]); dev_node.append([t.to(dev) for t in hn])
    out_pre = [torch.empty((T, D), dtype=tdt, device=dev) for _ in range(NL)]
    out_node = [torch.empty((M, D), dtype=tdt, device=dev) for _ in range(NL)]
    host_out_pre = [torch.empty((T, D), dtype=tdt).pin_memory() for _ in range(NL)]
    host_out_node = [torch.empty((M, D), dtype=tdt).pin_memory() for _ in range(NL)]

    def make_stack(flags_extra: int, params, n_slots=1 + M, max_tokens=T):
        layers = [upload_layer(p, w.cfg.act, md.MDRAFT_DT_SOFTPLUS | flags_extra, dev) for p in params]
        return DrafterStack(layers, n_slots, max_tokens, 1, max_tokens, 0, dev)

    # dispatch exactly as a user would: ask the library whether A has the power structure, then say so
    is_pow = all(md.mdraft_classify_A(upload_layer(p, w.cfg.act, 0, dev).A)[0] for p in w.params)
    stack = make_stack(md.MDRAFT_A_POWERS if is_pow else 0, w.params)
    stack_general = make_stack(0, w.params)

    cu = None  # one sequence of all T rows: the library needs no offsets for that
    slot0 = i32([0], dev)
    parent_slot = i32(np.where(w.tree.parents < 0, 0, w.tree.parents + 1), dev)
    node_slot = i32(np.arange(M) + 1, dev)
    levels = [int(v) for v in w.tree.level_offsets]
    acc_src = i32([w.accepted + 1], dev)

    def do_prefill(st, phase_events=None):
        st.prefill(dev_pre, out_pre, cu, T, None, slot0, None, phase_events)

    def do_tree(st):
        st.tree_round(dev_node, out_node, parent_slot, node_slot, levels)

    def do_commit(st):
        st.commit(acc_src, slot0)

    def step(st):
        do_prefill(st); do_tree(st); do_commit(st)

    # A drafting round is replayed from a CUDA graph, as the paper runs its drafter (Section 4.1): the library's calls
    # are stateless and take their indices from device memory, so one capture serves every step.
    def capture(fn):
        fn()  # the first call of anything happens outside the capture
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            fn()
        return g

    def time_graph(g, K, Wm):
        for _ in range(Wm):
            g.replay()
        barrier()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(K):
            g.replay()
        e1.record()
        barrier()
        return max_over_ranks(e0.elapsed_time(e1)) / K  # ms per replay

    K, Wm = args.steps, max(args.warmup, 3)
    g_step = capture(lambda: step(stack))
    sampler = ClockSampler(local)  # runs through every timed leg below (the headline loop alone lasts only tens of ms)
    sampler.start()
    time.sleep(0.3)                # nvidia-smi needs a moment before its first sample
    ms_step = time_graph(g_step, K, Wm)
    stack.check_status()
    Kp = min(K, 10)
    ms_prefill = time_graph(capture(lambda: do_prefill(stack)), Kp, 3)
    ms_tree = time_graph(capture(lambda: do_tree(stack)), Kp, 3)
    ms_commit = time_graph(capture(lambda: do_commit(stack)), Kp, 3)
    ms_step_general = time_graph(capture(lambda: step(stack_general)), Kp, 3)
    ms_prefill_general = time_graph(capture(lambda: do_prefill(stack_general)), Kp, 3)

    # ---- per-kernel split of the prefill call.  The three kernels of a call are launched eagerly with events between
    # them; a long spin kernel is queued first so that the host runs ahead and the events time the kernels, not the host.
    def kernel_split(st, reps):
        def ev():  # recorded once so that the underlying CUDA event exists before the library is handed its handle
            e = torch.cuda.Event(enable_timing=True)
            e.record()
            return e
        ks = [[], [], []]
        for _ in range(reps):
            evs = [[ev() for _ in range(4)] for _ in range(NL)]
            torch.cuda.synchronize()
            torch.cuda._sleep(40_000_000)  # about 20 ms at boost clock
            do_prefill(st, evs)
            torch.cuda.synchronize()
            for l in range(NL):
                for i in range(3):
                    ks[i].append(evs[l][i].elapsed_time(evs[l][i + 1]))
        return [1e3 * statistics.median(v) for v in ks]  # us: summary pass, carry scan, output pass

    split = kernel_split(stack, 3)
    split_general = kernel_split(stack_general, 2)

    # ---- tree step on the batched-serving shape (32 sequences x 32-node trees): whole round and its widest level
    bt = BatchedTree(seed=rank)
    bt_layers = [upload_layer(p, w.cfg.act, md.MDRAFT_DT_SOFTPLUS | (md.MDRAFT_A_POWERS if is_pow else 0), dev) for p in w.params]
    bt_cache = md.StateCache(NL, bt.S + bt.M, D, act=tdt, device=dev)
    bt_cache.ssm.normal_()
    bt_in = [[to_device(a, tdt).to(dev) for a in gen.node_inputs(bt.cfg, l, 0, bt.M)] for l in range(NL)]
    bt_out = [torch.empty((bt.M, D), dtype=tdt, device=dev) for _ in range(NL)]
    bt_par, bt_nod = i32(bt.parent, dev), i32(bt.nodes, dev)
    bt_status = torch.zeros(1, dtype=torch.int32, device=dev)
    lo, hi = bt.levels[-2], bt.levels[-1]

    def bt_round():
        for l in range(NL):
            md.mdraft_tree_step(bt_layers[l], bt_cache, l, *bt_in[l], bt_out[l], bt_par, bt_nod, bt.levels, bt_status)

    def bt_widest():
        for l in range(NL):
            md.mdraft_tree_step(bt_layers[l], bt_cache, l, *[a[lo:hi] for a in bt_in[l]], bt_out[l][lo:hi], bt_par[lo:hi], bt_nod[lo:hi],
                                None, bt_status)

    ms_bt_round = time_graph(capture(bt_round), Kp, 3)
    ms_bt_widest = time_graph(capture(bt_widest), Kp, 3)
    if int(bt_status.item()):
        raise RuntimeError("device status bits set in the batched tree leg")

    # ---- one tree level of the paper's widest kind (18 nodes, all children of the committed state) through the step
    # that forms dt, B and C itself, next to the split mode (conv step, torch matmuls, S6 step) and to the plain step
    # with dt, B, C given.  24 layers per replay, time per layer.
    PN, PR = 18, 48
    pj_W = [[to_device(a, tdt).to(dev) for a in gen.select_proj(w.cfg, l, PR)] for l in range(NL)]
    pj_Wt = [[a.T.contiguous() for a in ws_] for ws_ in pj_W]
    pj_in = [[a[:PN] for a in bt_in[l]] for l in range(NL)]
    pj_out, pj_u = torch.empty((PN, D), dtype=tdt, device=dev), torch.empty((PN, D), dtype=tdt, device=dev)
    pj_par, pj_nod = i32([0] * PN, dev), i32(list(range(1, PN + 1)), dev)
    fl = md.MDRAFT_DT_SOFTPLUS | (md.MDRAFT_A_POWERS if is_pow else 0)

    def pj_fused():
        for l in range(NL):
            md.mdraft_tree_step_proj(bt_layers[l], bt_cache, l, pj_W[l][0], pj_W[l][1], pj_in[l][0], pj_in[l][1], pj_out, pj_par, pj_nod, bt_status)

    def pj_split():
        for l in range(NL):
            md.mdraft_tree_step(bt_layers[l], bt_cache, l, pj_in[l][0], None, None, None, None, pj_u, pj_par, pj_nod, None, bt_status,
                                flags=md.MDRAFT_CONV_ONLY)
            s_ = pj_u @ pj_Wt[l][0]
            dt_ = (s_[:, :PR] @ pj_Wt[l][1]).contiguous()
            md.mdraft_tree_step(bt_layers[l], bt_cache, l, pj_u, pj_in[l][1], dt_, s_[:, PR:PR + 16].contiguous(), s_[:, PR + 16:].contiguous(),
                                pj_out, pj_par, pj_nod, None, bt_status, flags=fl | md.MDRAFT_PRECONV)

    def pj_plain():
        for l in range(NL):
            md.mdraft_tree_step(bt_layers[l], bt_cache, l, *pj_in[l], pj_out, pj_par, pj_nod, None, bt_status)

    proj_level = {"nodes": PN, "dt_rank": PR, "unit": "us per layer (CUDA-graph replay of 24 layers)",
                  "projection_step": time_graph(capture(pj_fused), Kp, 3) / NL * 1e3,
                  "split_mode": time_graph(capture(pj_split), Kp, 3) / NL * 1e3,
                  "plain_step_inputs_given": time_graph(capture(pj_plain), Kp, 3) / NL * 1e3}
    # wide levels: the projection step against the split mode, and what a caller following the header's width rule gets
    # (projection step up to MDRAFT_PROJ_STEP_MAX_NODES nodes per level, split mode beyond); 8 layers per replay
    if not args.quick:
        from paper_2506_01206_b200.drafter import PROJ_STEP_MAX_NODES
        NLw = 8
        wide = {}
        for PNw in (256, 442, 512, 1024):
            w_in = [[a[:PNw] for a in bt_in[l]] for l in range(NLw)]
            w_out, w_u = torch.empty((PNw, D), dtype=tdt, device=dev), torch.empty((PNw, D), dtype=tdt, device=dev)
            w_par, w_nod = i32([0] * PNw, dev), i32(list(range(1, PNw + 1)), dev)

            def w_fused():
                for l in range(NLw):
                    md.mdraft_tree_step_proj(bt_layers[l], bt_cache, l, pj_W[l][0], pj_W[l][1], w_in[l][0], w_in[l][1], w_out, w_par, w_nod, bt_status)

            def w_split():
                for l in range(NLw):
                    md.mdraft_tree_step(bt_layers[l], bt_cache, l, w_in[l][0], None, None, None, None, w_u, w_par, w_nod, None, bt_status,
                                        flags=md.MDRAFT_CONV_ONLY)
                    s_ = w_u @ pj_Wt[l][0]
                    dt_ = (s_[:, :PR] @ pj_Wt[l][1]).contiguous()
                    md.mdraft_tree_step(bt_layers[l], bt_cache, l, w_u, w_in[l][1], dt_, s_[:, PR:PR + 16].contiguous(), s_[:, PR + 16:].contiguous(),
                                        w_out, w_par, w_nod, None, bt_status, flags=fl | md.MDRAFT_PRECONV)

            tf_, ts_ = time_graph(capture(w_fused), Kp, 3) / NLw * 1e3, time_graph(capture(w_split), Kp, 3) / NLw * 1e3
            wide[str(PNw)] = {"projection_step": tf_, "split_mode": ts_, "by_width_rule": tf_ if PNw <= PROJ_STEP_MAX_NODES else ts_}
        proj_level["wide_levels_us_per_layer"] = wide
        proj_level["width_rule"] = "projection step up to %d nodes per level, split mode beyond (include/mdraft.h, drafter.PROJ_STEP_MAX_NODES)" % PROJ_STEP_MAX_NODES
    if int(bt_status.item()):
        raise RuntimeError("device status bits set in the projection leg")

    # ---- further prefill shapes (time per layer-call, CUDA-graph replay over distinct per-layer buffers that together
    # exceed L2): the long context, the packed batch and fp32 activations.  These legs time only; their inputs are drawn
    # on the device from the recipe's distributions (x, z, B, C ~ N(0,1), dt = clip(0.5 N(0,1))), the parity of these
    # shapes against the oracle is the business of tests/test_gpu_configs.py.
    def prefill_leg(act, lens, n_buf, reps):
        tdt_l = torch_act(act)
        es = 4 if act == "f32" else 2
        S_l, T_l = len(lens), int(sum(lens))
        gen_t = torch.Generator(device=dev); gen_t.manual_seed(1234 + rank)
        def rnd(shape, scale=1.0):
            return (torch.randn(shape, generator=gen_t, device=dev, dtype=torch.float32) * scale).to(tdt_l)
        bufs = []
        for _ in range(n_buf):
            dtv = rnd((T_l, D), 0.5).float().clamp_(float(gen.DT_PRE_LO), float(gen.DT_PRE_HI)).to(tdt_l)
            bufs.append([rnd((T_l, D)), rnd((T_l, D)), dtv, rnd((T_l, 16)), rnd((T_l, 16))])
        outs_l = [torch.empty((T_l, D), dtype=tdt_l, device=dev) for _ in range(n_buf)]
        lays = [upload_layer(w.params[l], act, md.MDRAFT_DT_SOFTPLUS | (md.MDRAFT_A_POWERS if is_pow else 0), dev) for l in range(n_buf)]
        st_l = DrafterStack(lays, S_l, T_l, S_l, max(lens), 0, dev)
        cu_l = None if S_l == 1 else i32(np.concatenate([[0], np.cumsum(lens)]), dev)
        slots_l = i32(np.arange(S_l), dev)
        fn = lambda: st_l.prefill(bufs, outs_l, cu_l, max(lens), None, slots_l)
        ms = time_graph(capture(fn), reps, 3) / n_buf
        st_l.check_status()
        bytes_l = 4 * es * T_l * D + 2 * 16 * es * T_l + S_l * (D * 16 * 4 + 3 * D * es)
        units = T_l * D
        del bufs, outs_l, st_l
        torch.cuda.empty_cache()
        return {"activations": act, "sequences": S_l, "tokens": T_l, "us_per_layer": ms * 1e3, "token_channels_per_s": units / (ms * 1e-3),
                "algorithmic_bytes_per_layer": bytes_l, "hbm_frac": bytes_l / (ms * 1e-3) / 1e9 / load_peaks()[0],
                "fp32_issue_frac_82_ops": ALU_LANE_OPS_PER_UNIT * units / (ms * 1e-3) / (SM_COUNT * FP32_LANES_PER_SM * SM_MAX_MHZ * 1e6),
                "fp32_issue_frac_70_ops": 70 * units / (ms * 1e-3) / (SM_COUNT * FP32_LANES_PER_SM * SM_MAX_MHZ * 1e6),
                "buffers": n_buf, "launches": md.mdraft_prefill_stack_launches(lays[0], n_buf, T_l, S_l, max(lens))}

    peak_hbm = load_peaks()[0]
    prefill_shapes = None
    if not args.quick:
        cfg4_lens = [int(v) for v in np.diff(gen.seq_lengths(gen.get_config(4)))]
        prefill_shapes = {
            "note": "whole prefill call (summary pass + carry scan + output pass) per layer; hbm_frac against the measured copy bandwidth; "
                    "fp32_issue_frac = lane-operations per token*channel (82 counted from the formulas the kernels evaluate, 70 a rounder estimate) x units / time / (148 x 128 x 1965 MHz)",
            "long_context_32768_bf16": prefill_leg("bf16", [32768], 4, 5),
            "packed_batch_32_seqs_1k_8k_bf16": prefill_leg("bf16", cfg4_lens, 2, 3),
            "fp32_activations_2048": prefill_leg("f32", [2048], 8, 10),
            "bf16_activations_2048_device_inputs": prefill_leg("bf16", [2048], 8, 10),
        }

    # ---- Mamba-2 (SSD) layer of the same size (24 heads of 64 channels, 128 states): context encode on the tensor cores
    # and the draft-tree step (memory-bound update of 786 KB states).  Inputs from the SSD recipe (host, seeded).
    roofline_ssd = None
    if not args.quick:
        from paper_2506_01206_b200.device_inputs import upload_ssd_layer
        SP, SN, NLs = 64, 128, 8
        scfg = gen.Config(97, "ssd-bench", NLs, D, SN, 4, "bf16", 1, (T, T), "none", 0, rank)
        s_lays = [upload_ssd_layer(gen.ssd_params(scfg, l, SP, SN), md.MDRAFT_DT_SOFTPLUS, dev) for l in range(NLs)]
        s_in = [[to_device(a, tdt).to(dev) for a in gen.ssd_inputs(scfg, l, 0, 0, T, SP, SN)] for l in range(NLs)]
        s_out = [torch.empty((T, D), dtype=tdt, device=dev) for _ in range(NLs)]
        s_nodes = 1 + M
        s_cache = md.StateCache(NLs, s_nodes, D, d_state=SN, act=tdt, device=dev)
        s_ws = torch.empty(md.mdraft_ssd_prefill_workspace_bytes(s_lays[0], T, 1), dtype=torch.uint8, device=dev)
        s_status = torch.zeros(1, dtype=torch.int32, device=dev)

        def ssd_prefill():
            for l in range(NLs):
                md.mdraft_ssd_prefill(s_lays[l], s_cache, l, *s_in[l], s_out[l], None, None, slot0, s_ws, s_status)

        s_nin = [[to_device(a, tdt).to(dev) for a in gen.ssd_inputs(scfg, l, 0, 1, M, SP, SN)] for l in range(NLs)]
        s_nout = [torch.empty((M, D), dtype=tdt, device=dev) for _ in range(NLs)]

        def ssd_tree():
            for l in range(NLs):
                md.mdraft_ssd_tree_step(s_lays[l], s_cache, l, *s_nin[l], s_nout[l], parent_slot, node_slot, levels, s_status)

        ms_sp = time_graph(capture(ssd_prefill), Kp, 3) / NLs
        ms_st = time_graph(capture(ssd_tree), Kp, 3) / NLs
        if int(s_status.item()):
            raise RuntimeError("device status bits set in the SSD leg")
        Hh = D // SP
        sp_bytes = 3 * T * D * 2 + T * Hh * 2 + 2 * T * SN * 2 + D * SN * 4 + 3 * D * 2
        n_chunks = -(-T // 128)
        # tensor-core work as issued: per (chunk, head) G 128x128x128, Y 128x64x128, C.H_in 128x64x128 twice (value and
        # remainder), state 128x64x128 twice; algorithmic: G once per chunk, no remainder products
        flops_issued = n_chunks * Hh * 2 * 128 * (128 * 128 + 64 * 128 + 2 * 64 * 128 + 2 * 64 * 128)
        flops_alg = n_chunks * 2 * 128 * 128 * 128 + n_chunks * Hh * 2 * 128 * (64 * 128 + 64 * 128 + 64 * 128)
        state_b = D * SN * 4 + 3 * D * 2
        st_bytes = M * (state_b + 2 * D * 2 + Hh * 2 + D * 2 + 2 * SN * 2) + len(set(int(v) for v in w.tree.parents)) * state_b
        try:
            tf_peak = float(json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))["bf16_tflops"])
        except Exception:
            tf_peak = 1590.0
        roofline_ssd = {
            "workload": "Mamba-2 (SSD) layer: %d tokens x %d channels = %d heads x 64, 128 states, bf16; %d distinct layers per replay" % (T, D, Hh, NLs),
            "prefill": {"bound": "hbm", "kernels": "ssd_chunk_state (tcgen05) + ssd_state_passing + ssd_chunk_scan (tcgen05)",
                        "us_per_layer": ms_sp * 1e3, "algorithmic_bytes_per_layer": sp_bytes,
                        "achieved": sp_bytes / (ms_sp * 1e-3) / 1e9, "peak": peak_hbm, "unit": "GB/s", "frac": sp_bytes / (ms_sp * 1e-3) / 1e9 / peak_hbm,
                        "tensor": {"issued_tflops": flops_issued / (ms_sp * 1e-3) / 1e12, "algorithmic_tflops": flops_alg / (ms_sp * 1e-3) / 1e12,
                                   "peak": tf_peak, "frac_issued": flops_issued / (ms_sp * 1e-3) / 1e12 / tf_peak},
                        "token_channels_per_s": T * D / (ms_sp * 1e-3),
                        "note": "HBM binds before the tensor cores at this shape (20.8 MB against 2.9 GFLOP per layer); the kernels are "
                                "far from either: blocks of 256 threads, three to an SM, walk phases that wait for one another"},
            "tree_step": {"bound": "hbm", "kernel": "ssd_step_kernel", "nodes": M, "levels": len(levels) - 1, "us_per_layer_round": ms_st * 1e3,
                          "algorithmic_bytes_per_layer_round": st_bytes, "achieved": st_bytes / (ms_st * 1e-3) / 1e9, "peak": peak_hbm, "unit": "GB/s",
                          "frac": st_bytes / (ms_st * 1e-3) / 1e9 / peak_hbm, "node_updates_per_s": M / (ms_st * 1e-3)},
        }
        del s_in, s_out, s_cache, s_nin, s_nout
        torch.cuda.empty_cache()
    clocks = sampler.stop()

    # ---- end to end: pinned host inputs -> device -> the path -> outputs back to the host, every step, through the
    # public calls with their stream argument: three streams, so that layer l+1's inputs travel while layer l computes
    # and layer l-1's outputs leave.  (The launches are eager here: each layer's calls wait on that layer's copy.)
    s_in, s_comp, s_out = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.Stream()
    ev_in = [torch.cuda.Event() for _ in range(NL)]
    ev_comp = [torch.cuda.Event() for _ in range(NL)]
    ev_out = [torch.cuda.Event() for _ in range(NL)]
    e2e_state = {"first": True}

    def e2e_step():
        first = e2e_state["first"]
        for l in range(NL):
            with torch.cuda.stream(s_in):
                if not first:
                    s_in.wait_event(ev_comp[l])      # the previous step has finished reading this layer's inputs
                for d_t, h_t in zip(dev_pre[l] + dev_node[l], host_pre[l] + host_node[l]):
                    d_t.copy_(h_t, non_blocking=True)
                ev_in[l].record(s_in)
            with torch.cuda.stream(s_comp):
                s_comp.wait_event(ev_in[l])
                if not first:
                    s_comp.wait_event(ev_out[l])     # the previous step's outputs of this layer have left
                stack.prefill(dev_pre, out_pre, cu, T, None, slot0, s_comp, None, [l])
                stack.tree_round(dev_node, out_node, parent_slot, node_slot, levels, s_comp, [l])
                ev_comp[l].record(s_comp)
            with torch.cuda.stream(s_out):
                s_out.wait_event(ev_comp[l])
                host_out_pre[l].copy_(out_pre[l], non_blocking=True)
                host_out_node[l].copy_(out_node[l], non_blocking=True)
                ev_out[l].record(s_out)
        with torch.cuda.stream(s_comp):
            stack.commit(acc_src, slot0, s_comp)
        e2e_state["first"] = False

    def e2e_join():
        cur = torch.cuda.current_stream()
        done = torch.cuda.Event()
        for st in (s_in, s_comp, s_out):
            done.record(st)
            cur.wait_event(done)

    Ke = min(K, 5)
    for _ in range(2):
        e2e_step()
    e2e_join()
    barrier()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for st in (s_in, s_comp, s_out):
        st.wait_event(e0)
    for _ in range(Ke):
        e2e_step()
    e2e_join()
    e1.record()
    barrier()
    stack.check_status()
    ms_e2e = max_over_ranks(e0.elapsed_time(e1)) / Ke
    h2d = sum(t.numel() * t.element_size() for l in range(NL) for t in host_pre[l] + host_node[l])
    d2h = sum(t.numel() * t.element_size() for l in range(NL) for t in (host_out_pre[l], host_out_node[l]))

    units_step = NL * T * D                      # prefill token*channels per step per GPU
    node_updates = NL * M
    value = replicas.whole_job_throughput(units_step, ms_step, world)
    peak, peak_src = load_peaks()
    # one launch takes all layers (up to 32) of the encode, or of a tree level
    launches = md.mdraft_prefill_stack_launches(stack.layers[0], NL, T, 1, T) + -(-NL // 32) * (len(levels) - 1) + 1
    alu_peak = SM_COUNT * FP32_LANES_PER_SM * SM_MAX_MHZ * 1e6  # fp32 lane-ops/s at the maximum SM clock

    # dominant kernel: the output pass of the prefill (chunk_kernel<bf16, kOut>), which takes all layers of the step's encode in
    # one launch: every sequence is left whole, so it is the call's only kernel.  The three kernels of a call for one
    # layer, which is cut into chunks, are quoted beside it.
    pb = w.prefill_bytes_per_layer()
    if md.mdraft_prefill_stack_launches(stack.layers[0], NL, T, 1, T) != 1:
        raise RuntimeError("the step's encode is expected to be one launch")
    scan_s = call_s = ms_prefill * 1e-3 / NL
    kname = "chunk_kernel<bf16, 256-channel blocks, %s, output pass>" % ("structured A" if is_pow else "general A")
    lane_ops = ALU_LANE_OPS_PER_UNIT * T * D
    roofline = {
        # bf16 activations: 82 fp32 lane-ops against 8 bytes per token*channel put this kernel's ridge point far on
        # the arithmetic side of the machine balance (37.2 T lane-op/s against 6.5 TB/s = 5.7 lane-ops per byte), so
        # the bound that applies is the fp32 issue rate; the HBM figure is kept beside it.
        "bound": "alu", "kernel": kname, "achieved": lane_ops / scan_s / 1e12, "peak": alu_peak / 1e12,
        "unit": "T fp32 lane-op/s (one instruction on one lane; an FMA counts once)", "frac": lane_ops / scan_s / alu_peak,
        "traffic": ncu_traffic("prefill_output_pass")[0], "traffic_kernel": ncu_traffic("prefill_output_pass")[1],
        "peak_source": "148 SMs x 128 fp32 lanes x %.0f MHz (clocks.max.sm)" % SM_MAX_MHZ,
        "algorithmic_lane_ops_per_launch": NL * lane_ops, "algorithmic_bytes_per_launch": NL * pb, "launch_us": 1e3 * ms_prefill,
        "timed": "CUDA-graph replay of the step's own encode call: one launch of this kernel over the 24 layers",
        "hbm": {"achieved": pb / scan_s / 1e9, "peak": peak, "unit": "GB/s", "frac": pb / scan_s / 1e9 / peak, "peak_source": peak_src,
                "frac_of_nominal_8000": pb / scan_s / 1e9 / 8000.0},
        "whole_prefill_call": {"us": call_s * 1e6, "achieved": pb / call_s / 1e9, "frac": pb / call_s / 1e9 / peak,
                               "alu_frac": lane_ops / call_s / alu_peak,
                               "summary_pass_us": split[0], "carry_scan_us": split[1], "output_pass_us": split[2],
                               "timed": "call: CUDA-graph replay of the call over 24 layers, time / 24; the *_pass_us / carry_scan_us keys: the three kernels of a call for ONE layer (cut into chunks), CUDA events recorded by the library between them, launched eagerly with the host queued ahead (no overlap between the kernels, event gaps included)"},
    }
    tb = w.tree_bytes_per_layer()
    bt_round_bytes = sum(bt.level_bytes(a, b) for a, b in zip(bt.levels[:-1], bt.levels[1:]))
    bt_wide_bytes = bt.level_bytes(lo, hi)
    roofline_tree = {
        "bound": "hbm", "kernel": "tree_step_kernel<bf16>", "workload": "32 sequences x 32-node trees, widest level (%d nodes), 24 layers" % (hi - lo),
        "achieved": NL * bt_wide_bytes / (ms_bt_widest * 1e-3) / 1e9, "peak": peak, "unit": "GB/s",
        "frac": NL * bt_wide_bytes / (ms_bt_widest * 1e-3) / 1e9 / peak, "traffic": ncu_traffic("tree_step_widest_level")[0], "traffic_kernel": ncu_traffic("tree_step_widest_level")[1],
        "algorithmic_bytes_per_launch": NL * bt_wide_bytes, "launch_us": 1e3 * ms_bt_widest,
        "timed": "CUDA-graph replay of the level, one launch over the 24 layers (distinct 110 MB pools)",
        "whole_round": {"ms": ms_bt_round, "levels": [b - a for a, b in zip(bt.levels[:-1], bt.levels[1:])],
                        "node_updates_per_s": world * NL * bt.M / (ms_bt_round * 1e-3),
                        "hbm_frac": NL * bt_round_bytes / (ms_bt_round * 1e-3) / 1e9 / peak},
    }
    extra = {
        "prefill": {"value": world * units_step / (ms_prefill * 1e-3), "unit": UNIT, "ms": ms_prefill,
                    "hbm_frac": NL * pb / (ms_prefill * 1e-3) / 1e9 / peak},
        "tree_step": {"value": world * node_updates / (ms_tree * 1e-3), "unit": "node-updates/s", "ms": ms_tree,
                      "nodes": M, "levels": len(levels) - 1, "algorithmic_bytes_per_layer": tb,
                      "hbm_frac": NL * tb / (ms_tree * 1e-3) / 1e9 / peak,
                      "note": "levels of 1-64 nodes at batch 1: every launch is a chain of dependent memory round trips"},
        "commit": {"ms": ms_commit, "hbm_frac": w.commit_bytes() / (ms_commit * 1e-3) / 1e9 / peak},
    }
    general = {
        "value": world * units_step / (ms_step_general * 1e-3), "ms_per_step": ms_step_general, "prefill_ms": ms_prefill_general,
        "summary_pass_us": split_general[0], "carry_scan_us": split_general[1], "output_pass_us": split_general[2],
        "hbm_frac_output_pass": pb / (split_general[2] * 1e-6) / 1e9 / peak,
        "note": "same workload with the A_POWERS hint withheld: one exponential per (token, channel, state)",
    }

    # ---- context figure: drafting latency per round of a whole 130M-shaped block stack with real data dependence (random
    # weights, one CUDA graph per generation step), the quantity of the paper's Table 4.  Not part of `value`.  With bf16
    # weights and levels of at most 64 nodes a generation runs in the library's block kernels whichever mode was asked for;
    # the modes themselves (split: conv step -> torch matmuls for the projections -> S6 step; projection step: one
    # launch does all of that) are what other types and wider levels run, and are timed with the block kernels off.
    drafter = None
    if rank == 0 and world == 1:
        from paper_2506_01206_b200.drafter import ToyDrafter
        drafter = {"unit": "ms per draft round (host launches and top-k between generation steps included)",
                   "paper_context": "6.62 (chain of 5) and 8.30 (tree (3,2,2,1,1)) on an RTX 4090, unit unstated, Mamba-130M drafter (paper Table 4)"}

        def round_ms(fn):
            for _ in range(3):
                fn()
            torch.cuda.synchronize()
            ts = []
            for _ in range(10):
                t0 = time.perf_counter()
                fn()
                torch.cuda.synchronize()
                ts.append((time.perf_counter() - t0) * 1e3)
            return statistics.median(ts)

        for mode, fused, block in (("block_kernels", False, True), ("split_mode", False, False), ("projection_step", True, False)):
            td = ToyDrafter(max_nodes=64, seed=0, device=dev, fused=fused)
            td.block_kernels = td.block_kernels and block
            drafter[mode] = {}
            for name, cfg_t in (("chain_5", (1, 1, 1, 1, 1)), ("tree_3_2_2_1_1", (3, 2, 2, 1, 1))):
                drafter[mode][name] = round_ms(lambda: td.draft_round(11, cfg_t))
                if block:   # the same round as one replayed graph (one host launch per round)
                    drafter.setdefault("block_kernels_one_graph_per_round", {})[name] = round_ms(lambda: td.draft_round_one_graph(11, cfg_t))
            if int(td.status.item()):
                raise RuntimeError("device status bits set in the drafter leg")
            del td

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu:
        cores = os.cpu_count() or 1
        reps, total, used = 0, 0.0, cores
        while total < 10.0 and reps < 64:   # whole steps of the oracle until about 10 s of work are on the clock
            _, dt, used = time_oracle_sample(w, NL, cores)
            total += dt; reps += 1
        v1, dt1, _ = time_oracle_sample(w, 2, 1)   # the same oracle on one thread, two layers of the step
        cpu = {"value": reps * units_step / total, "unit": UNIT, "cores": used, "kind": "oracle", "seconds": total,
               "single_thread": {"value": v1, "unit": UNIT, "seconds": dt1, "sample": "2 of the 24 layers of one step, one thread"},
               "sample": "%d repetitions of the whole step (24 layers: prefill 2048 tokens + 150-node tree path by path + commit), fp64" % reps}

    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": K, "warmup": Wm,
            "ms_per_step": ms_step, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32", "data": "synthetic",
            "config": {"workload": WORKLOAD, "activations": "bf16", "state": "fp32", "n_layers": NL, "tokens": T, "d_inner": D,
                       "d_state": 16, "tree_nodes": M, "tree_levels": len(levels) - 1,
                       "a_mode": "powers (A[d][n]=(n+1)A[d][0] verified on the device at set-up)" if is_pow else "general",
                       "launch": "one CUDA graph per step (prefill of 24 layers, 6-level draft round, commit), replayed",
                       "l2": "inputs larger than L2: each step streams 24 layers of distinct buffers (0.61 GB) plus a 0.39 GB state pool",
                       "replicas": "independent per GPU (no exchange step on this path)"},
            "clocks": clocks,
            "e2e": {"value": world * units_step / (ms_e2e * 1e-3), "unit": UNIT, "ms_per_step": ms_e2e,
                    "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h, "steps": Ke},
            "gpu_launches": launches * K,
            "gpu_launches_per_step": launches,
            "roofline": roofline,
            "roofline_tree_step": roofline_tree,
            "phases": extra,
            "general_A": general,
            "prefill_shapes": prefill_shapes,
            "roofline_ssd": roofline_ssd,
            "projection_level": proj_level,
            "drafter_round": drafter,
            "cpu_baseline": cpu,
        }
        print(json.dumps(line))
    replicas.finish(world)


# ----------------------------------------------------------------------------------------------- profiler cases
def profile_case(what, sizes):
    """Small, self-contained runs of one kernel family for a profiler (ncu): few launches, well under 1 GB on the device,
    inputs larger than L2 across the layers so that DRAM counters still mean something.
      prefill [tokens=2048] [layers=4] [reps=3] [fp32=0] [general=0]   130M-shaped context encode layer by layer, bf16 (or fp32) activations
      stack   [tokens=2048] [layers=24] [reps=3]           the same, all layers in one call
      tree    [layers=4] [reps=2]                          one batched-serving draft round, 32 sequences x 32-node trees
      proj    [nodes=18] [layers=24] [reps=3]              one tree level through the step that forms dt, B, C itself
      ssd     [tokens=2048] [layers=2] [reps=3]            Mamba-2 (SSD) context encode, 24 heads x 64 channels, 128 states
      generation [nodes=18] [layers=24] [reps=3]           one generation of the drafter's block stack"""
    import torch
    import paper_2506_01206_b200 as md
    from paper_2506_01206_b200.device_inputs import i32, to_device, torch_act, upload_layer
    flags = md.MDRAFT_DT_SOFTPLUS | md.MDRAFT_A_POWERS
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    if what == "prefill":
        tokens, n_layers, reps, fp32, general = (list(sizes) + [2048, 4, 3, 0, 0][len(sizes):])[:5]
        cfg = gen.get_config(1)
        act = "f32" if fp32 else cfg.act
        tdt, D = torch_act(act), cfg.d_inner
        lays = [upload_layer(gen.layer_params(cfg, l), act, md.MDRAFT_DT_SOFTPLUS if general else flags) for l in range(n_layers)]
        ins = [[to_device(a, tdt) for a in gen.prefill_inputs(cfg, l, tokens)] for l in range(n_layers)]
        outs = [torch.empty((tokens, D), dtype=tdt, device="cuda") for _ in range(n_layers)]
        cache = md.StateCache(n_layers, 1, D, act=tdt)
        ws = torch.empty(max(256, md.mdraft_prefill_workspace_bytes(lays[0], tokens, 1, tokens)), dtype=torch.uint8, device="cuda")
        slot = i32([0])
        for _ in range(reps):
            for l in range(n_layers):
                md.mdraft_conv_scan_prefill(lays[l], cache, l, *ins[l], outs[l], None, tokens, None, slot, ws, 0, status)
        torch.cuda.synchronize()
        print("prefill: %d tokens x %d channels, %s, %d layers x %d, status %d" % (tokens, D, act, n_layers, reps, int(status.item())))
    elif what == "stack":
        from paper_2506_01206_b200.stack import DrafterStack
        tokens, n_layers, reps = (list(sizes) + [2048, 24, 3][len(sizes):])[:3]
        cfg = gen.get_config(1)
        tdt, D = torch_act(cfg.act), cfg.d_inner
        st = DrafterStack([upload_layer(gen.layer_params(cfg, l), cfg.act, flags) for l in range(n_layers)], 1, tokens, 1, tokens)
        ins = [[to_device(a, tdt) for a in gen.prefill_inputs(cfg, l, tokens)] for l in range(n_layers)]
        outs = [torch.empty((tokens, D), dtype=tdt, device="cuda") for _ in range(n_layers)]
        for _ in range(reps):
            st.prefill(ins, outs, None, tokens, None, i32([0]))
        torch.cuda.synchronize()
        st.check_status()
        print("stack: %d tokens x %d channels, %d layers in one call x %d" % (tokens, D, n_layers, reps))
    elif what == "generation":
        from paper_2506_01206_b200.drafter import ToyDrafter
        n_nodes, n_layers, reps = (list(sizes) + [18, 24, 3][len(sizes):])[:3]
        td = ToyDrafter(n_layers=n_layers, max_nodes=n_nodes)
        td.node_slot.copy_(i32(list(range(1, n_nodes + 1))))
        for _ in range(reps):
            td.generation(0, n_nodes, use_graph=False)
        torch.cuda.synchronize()
        print("generation: %d nodes, %d layers x %d, status %d" % (n_nodes, n_layers, reps, int(td.status.item())))
    elif what == "tree":
        n_layers, reps = (list(sizes) + [4, 2][len(sizes):])[:2]
        bt = BatchedTree(seed=0)
        cfg, D = bt.cfg, bt.cfg.d_inner
        tdt = torch_act(cfg.act)
        lays = [upload_layer(gen.layer_params(cfg, l), cfg.act, flags) for l in range(n_layers)]
        ins = [[to_device(a, tdt) for a in gen.node_inputs(cfg, l, 0, bt.M)] for l in range(n_layers)]
        outs = [torch.empty((bt.M, D), dtype=tdt, device="cuda") for _ in range(n_layers)]
        cache = md.StateCache(n_layers, bt.S + bt.M, D, act=tdt)
        cache.ssm.normal_()
        par, nod = i32(bt.parent), i32(bt.nodes)
        for _ in range(reps):   # every level of all layers in one launch, as the round runs
            if not md.mdraft_tree_step_stack(lays, range(n_layers), cache, ins, outs, par, nod, bt.levels, status):
                raise RuntimeError("the layers did not run side by side")
        torch.cuda.synchronize()
        print("tree: %d nodes, levels %s, %d layers x %d, status %d" % (bt.M, np.diff(bt.levels).tolist(), n_layers, reps, int(status.item())))
    elif what == "ssd":
        from paper_2506_01206_b200.device_inputs import upload_ssd_layer
        tokens, n_layers, reps = (list(sizes) + [2048, 2, 3][len(sizes):])[:3]
        D, P, N = 1536, 64, 128
        cfg = gen.Config(97, "ssd-profile", n_layers, D, N, 4, "bf16", 1, (tokens, tokens), "none", 0, 0)
        tdt = torch.bfloat16
        lays = [upload_ssd_layer(gen.ssd_params(cfg, l, P, N)) for l in range(n_layers)]
        ins = [[to_device(a, tdt) for a in gen.ssd_inputs(cfg, l, 0, 0, tokens, P, N)] for l in range(n_layers)]
        outs = [torch.empty((tokens, D), dtype=tdt, device="cuda") for _ in range(n_layers)]
        cache = md.StateCache(n_layers, 1, D, d_state=N, act=tdt)
        ws = torch.empty(md.mdraft_ssd_prefill_workspace_bytes(lays[0], tokens, 1), dtype=torch.uint8, device="cuda")
        slot = i32([0])
        for _ in range(reps):
            for l in range(n_layers):
                md.mdraft_ssd_prefill(lays[l], cache, l, *ins[l], outs[l], None, None, slot, ws, status)
        torch.cuda.synchronize()
        print("ssd: %d tokens x %d channels (%d heads), %d layers x %d, status %d" % (tokens, D, D // P, n_layers, reps, int(status.item())))
    else:
        n_nodes, n_layers, reps = (list(sizes) + [18, 24, 3][len(sizes):])[:3]
        dt_rank = 48
        cfg = gen.get_config(1)
        tdt, D = torch_act(cfg.act), cfg.d_inner
        lays = [upload_layer(gen.layer_params(cfg, l), cfg.act, flags) for l in range(n_layers)]
        Ws = [[to_device(v, tdt) for v in gen.select_proj(cfg, l, dt_rank)] for l in range(n_layers)]
        ins = [[to_device(a, tdt) for a in gen.node_inputs(cfg, l, 0, n_nodes)[:2]] for l in range(n_layers)]
        out = torch.empty((n_nodes, D), dtype=tdt, device="cuda")
        cache = md.StateCache(n_layers, 1 + n_nodes, D, act=tdt)
        cache.ssm.normal_(); cache.conv.normal_()
        par, nod = i32([0] * n_nodes), i32(list(range(1, n_nodes + 1)))
        for _ in range(reps):
            for l in range(n_layers):
                md.mdraft_tree_step_proj(lays[l], cache, l, Ws[l][0], Ws[l][1], ins[l][0], ins[l][1], out, par, nod, status)
        torch.cuda.synchronize()
        print("proj: %d nodes x %d channels, dt_rank %d, %d layers x %d, status %d" % (n_nodes, D, dt_rank, n_layers, reps, int(status.item())))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu", action="store_true", help="skip the CPU-oracle baseline leg")
    ap.add_argument("--quick", action="store_true", help="skip the further prefill shapes (long context, packed batch, fp32)")
    ap.add_argument("--profile-case", choices=["prefill", "stack", "tree", "proj", "ssd", "generation"], help="run one small kernel case for a profiler and exit")
    ap.add_argument("sizes", nargs="*", type=int, help="sizes of the profile case (see profile_case)")
    args = ap.parse_args()
    if args.profile_case:
        profile_case(args.profile_case, args.sizes)
    elif args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
