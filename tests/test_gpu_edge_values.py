"""Inputs OUTSIDE the benchmark's recipe, through every kernel, against the fp64 oracle.

The recipe keeps the step size inside [1e-3, 1e-1] and A at -(1..16), so on those inputs some branches of the
kernels never run: the large-argument shortcut of softplus, decays that underflow (and the clamp of the
polynomial exponential at 2^-126), the power chain of a structured A once r^16 flushes to zero, A = 0 (the
cumulative-sum case), a step size of exactly 0 (the frozen-state case) and steep A rows.  A trained drafter does
not stay inside the recipe; these cases are the closed-form cases of the recurrence, run through the kernels:

  big_dt  : pre-activations from -90 to +45 under softplus (step sizes from 0 to 45)
  zero_dt : step size given as such (no softplus), a mixture of exact zeros and small positive values
  A_zero  : channels (and single states) whose A is exactly 0
  A_steep : A rows from -12.5 down to -200
"""

import numpy as np
import pytest
import torch

import gen
import oracle
import parity
from parity import TOL, TOL_STATE, assert_close
from test_gpu_parity_small import run_gpu_prefill, run_oracle_prefill
from test_gpu_prefill_cluster import form
from test_gpu_tree import TreeRig
from test_gpu_tree_proj import ProjRig

pytestmark = pytest.mark.gpu

import paper_2506_01206_b200 as md
from paper_2506_01206_b200.device_inputs import to_device, upload_layer

REGIMES = ["big_dt", "zero_dt", "A_zero", "A_steep"]


def case_seed(regime, act, powers, kernel):
    return 1000 * kernel + 16 * REGIMES.index(regime) + 2 * (act == "bf16") + int(powers)


def shape_A(params, regime, powers, g):
    """Overwrites params.A for the regime; with ``powers`` the result keeps A[d][n] == (n+1) A[d][0] exactly in fp32."""
    Dn, N = params.A.shape
    n1 = np.arange(1, N + 1, dtype=np.float32)
    if regime == "A_steep":
        if powers:
            a0 = g.choice(np.array([-12.5, -2.5, -40.0], dtype=np.float32), size=Dn)
            params.A[:] = a0[:, None] * n1[None, :]
        else:
            params.A[:] = -g.uniform(40.0, 200.0, size=(Dn, N)).astype(np.float32)
    elif regime == "A_zero":
        if powers:
            a0 = np.where(np.arange(Dn) % 3 == 0, 0.0, -1.0).astype(np.float32)
            params.A[:] = a0[:, None] * n1[None, :]
        else:
            params.A[np.arange(Dn) % 3 == 0, :] = 0.0     # whole channels: a running sum of the inputs
            params.A[:, ::4] = np.where(g.random((Dn, N // 4)) < 0.5, 0.0, params.A[:, ::4])  # and single states
    elif powers:
        params.A[:] = -np.tile(n1, (Dn, 1))


def shape_dt(dt, params, regime, act, g):
    """Returns the dt array for the regime (values representable in ``act``) and sets the bias; True if the step
    size is to be taken as given (no softplus)."""
    if regime == "big_dt":
        kind = g.integers(0, 4, size=dt.shape)
        v = np.where(kind == 0, g.normal(-4.6, 0.5, size=dt.shape),
                     np.where(kind == 1, g.uniform(15.0, 45.0, size=dt.shape),
                              np.where(kind == 2, g.uniform(-90.0, -20.0, size=dt.shape), g.uniform(-3.0, 3.0, size=dt.shape))))
        params.dt_bias[:] = g.uniform(-0.5, 0.5, size=params.dt_bias.shape).astype(np.float32)
        return gen.round_to_act(v.astype(np.float32), act), False
    if regime == "zero_dt":
        v = np.where(g.random(dt.shape) < 0.5, 0.0, g.uniform(0.001, 0.2, size=dt.shape))
        params.dt_bias[:] = 0.0
        return gen.round_to_act(v.astype(np.float32), act), True
    return dt, False


def flags_for(raw_step, powers):
    return (0 if raw_step else md.MDRAFT_DT_SOFTPLUS) | (md.MDRAFT_A_POWERS if powers else 0)


@pytest.mark.parametrize("regime", REGIMES)
@pytest.mark.parametrize("act", ["f32", "bf16"])
@pytest.mark.parametrize("powers", [False, True])
def test_prefill_outside_the_recipe(regime, act, powers):
    g = np.random.default_rng(case_seed(regime, act, powers, 0))
    lens = [150, 3, 77]
    cfg = parity.small_config(200, act, len(lens), cid=93)
    prob = parity.make_problem(cfg, lens, conv_bias=True, general_A=not powers)
    shape_A(prob.params, regime, powers, g)
    prob.dt, raw = shape_dt(prob.dt, prob.params, regime, act, g)
    flags = flags_for(raw, powers)
    if powers:
        assert md.mdraft_classify_A(upload_layer(prob.params, act, flags).A)[0], "the test's A must have the promised structure"
    h0 = g.normal(size=(len(lens), 200, 16)).astype(np.float32)
    c0 = gen.round_to_act(g.normal(size=(len(lens), 3, 200)).astype(np.float32), act)
    o_out, o_conv, o_h = run_oracle_prefill(prob, flags, c0, h0)
    for chunk_len in (32, 4096):   # split into chunks (summary pass + carry scan) and whole
        g_out, g_conv, g_h = run_gpu_prefill(prob, flags, chunk_len, c0, h0)
        assert_close(g_out, o_out, TOL[act], f"out, chunk_len {chunk_len}")
        assert_close(g_h, o_h, TOL_STATE, f"final SSM state, chunk_len {chunk_len}")
        assert np.array_equal(g_conv, o_conv)


@pytest.mark.parametrize("regime", [r for r in REGIMES if r != "zero_dt"])   # the one-kernel form forms its step sizes by softplus
@pytest.mark.parametrize("act", ["f32", "bf16"])
@pytest.mark.parametrize("powers", [False, True])
def test_one_kernel_prefill_outside_the_recipe(regime, act, powers):
    g = np.random.default_rng(case_seed(regime, act, powers, 3))
    for lens, have_state in (([150], True), ([150, 3, 77], False)):
        prob = parity.make_problem(parity.small_config(200, act, len(lens), cid=93), lens, conv_bias=True, general_A=not powers)
        shape_A(prob.params, regime, powers, g)
        prob.dt, raw = shape_dt(prob.dt, prob.params, regime, act, g)
        assert not raw
        flags = flags_for(False, powers)
        lay = upload_layer(prob.params, act, flags)
        assert not powers or md.mdraft_classify_A(lay.A)[0], "the test's A must have the promised structure"
        assert form(lay, 1, lens) != (0, 0)
        h0, c0 = (g.normal(size=(1, 200, 16)).astype(np.float32), gen.round_to_act(g.normal(size=(1, 3, 200)).astype(np.float32), act)) if have_state else (None, None)
        o_out, o_conv, o_h = run_oracle_prefill(prob, flags, c0, h0)
        g_out, g_conv, g_h = run_gpu_prefill(prob, flags, 0, c0, h0)
        assert_close(g_out, o_out, TOL[act], f"out, lengths {lens}")
        assert_close(g_h, o_h, TOL_STATE, f"final SSM state, lengths {lens}")
        assert np.array_equal(g_conv, o_conv)


@pytest.mark.parametrize("act", ["f32", "bf16"])
@pytest.mark.parametrize("powers", [False, True])
def test_one_kernel_prefill_whose_softplus_underflows_leaves_the_state_bit_identical(act, powers):
    """log(1 + exp(-200)) is 0 in fp32: the folds of the chunks' summaries give back what the slot held."""
    g = np.random.default_rng(18)
    prob = parity.make_problem(parity.small_config(136, act, 1, cid=93), [90], conv_bias=True, general_A=not powers)
    shape_A(prob.params, "", powers, g)
    prob.dt = gen.round_to_act(g.normal(size=prob.dt.shape).astype(np.float32), act)
    prob.params.dt_bias[:] = -200.0
    flags = flags_for(False, powers)
    assert form(upload_layer(prob.params, act, flags), 1, [90]) != (0, 0)
    h0 = g.normal(size=(1, 136, 16)).astype(np.float32)
    c0 = gen.round_to_act(g.normal(size=(1, 3, 136)).astype(np.float32), act)
    g_out, _, g_h = run_gpu_prefill(prob, flags, 0, c0, h0)
    assert np.array_equal(g_h.astype(np.float32).view(np.uint32), h0.view(np.uint32)), "a zero step size must freeze the state exactly"
    o_out, _, _ = run_oracle_prefill(prob, flags, c0, h0)
    assert_close(g_out, o_out, TOL[act], "out = (C.h0 + D u) * SiLU(z)")


@pytest.mark.parametrize("act", ["f32", "bf16"])
@pytest.mark.parametrize("powers", [False, True])
@pytest.mark.parametrize("chunk_len", [16, 4096])
def test_prefill_with_zero_step_size_leaves_the_state_bit_identical(act, powers, chunk_len):
    """Delta = 0 at every token: exp(0 * A) = 1 and the input term vanishes, so the state written to the final slot
    is, bit for bit, the state read from the starting slot, through the chunk summaries and the carry scan too."""
    g = np.random.default_rng(17)
    lens = [90, 41]
    cfg = parity.small_config(136, act, len(lens), cid=93)
    prob = parity.make_problem(cfg, lens, conv_bias=True, general_A=not powers)
    shape_A(prob.params, "", powers, g)
    prob.dt = np.zeros_like(prob.dt)
    prob.params.dt_bias[:] = 0.0
    flags = flags_for(True, powers)
    h0 = g.normal(size=(len(lens), 136, 16)).astype(np.float32)
    c0 = gen.round_to_act(g.normal(size=(len(lens), 3, 136)).astype(np.float32), act)
    g_out, _, g_h = run_gpu_prefill(prob, flags, chunk_len, c0, h0)
    assert np.array_equal(g_h.astype(np.float32).view(np.uint32), h0.view(np.uint32)), "a zero step size must freeze the state exactly"
    o_out, _, o_h = run_oracle_prefill(prob, flags, c0, h0)
    assert np.array_equal(o_h, h0.astype(np.float64))
    assert_close(g_out, o_out, TOL[act], "out = (C.h0 + D u) * SiLU(z)")


@pytest.mark.parametrize("act", ["f32", "bf16"])
@pytest.mark.parametrize("powers", [False, True])
@pytest.mark.parametrize("chunk_len", [16, 4096])
def test_prefill_whose_softplus_underflows_leaves_the_state_bit_identical(act, powers, chunk_len):
    """The same with the step size from softplus: log(1 + exp(-200)) is 0 in fp32."""
    g = np.random.default_rng(18)
    lens = [90, 41]
    cfg = parity.small_config(136, act, len(lens), cid=93)
    prob = parity.make_problem(cfg, lens, conv_bias=True, general_A=not powers)
    shape_A(prob.params, "", powers, g)
    prob.dt = gen.round_to_act(g.normal(size=prob.dt.shape).astype(np.float32), act)
    prob.params.dt_bias[:] = -200.0
    flags = flags_for(False, powers)
    h0 = g.normal(size=(len(lens), 136, 16)).astype(np.float32)
    c0 = gen.round_to_act(g.normal(size=(len(lens), 3, 136)).astype(np.float32), act)
    g_out, _, g_h = run_gpu_prefill(prob, flags, chunk_len, c0, h0)
    assert np.array_equal(g_h.astype(np.float32).view(np.uint32), h0.view(np.uint32)), "a zero step size must freeze the state exactly"
    o_out, _, _ = run_oracle_prefill(prob, flags, c0, h0)
    assert_close(g_out, o_out, TOL[act], "out = (C.h0 + D u) * SiLU(z)")


@pytest.mark.parametrize("act", ["f32", "bf16"])
@pytest.mark.parametrize("powers", [False, True])
def test_prefill_in_pieces_is_the_whole_bit_for_bit(act, powers):
    """A state that goes through a slot between two unsplit calls is the state that stays in registers."""
    cfg = parity.small_config(136, act, 1, cid=93)
    prob = parity.make_problem(cfg, [160], conv_bias=True, general_A=not powers)
    flags = flags_for(False, powers)
    whole = run_gpu_prefill(prob, flags, 4096)
    outs, conv, h = [], None, None
    for lo, hi in ((0, 48), (48, 160)):
        piece = parity.make_problem(cfg, [hi - lo], conv_bias=True, general_A=not powers)
        piece.params = prob.params
        for name in ("x", "z", "dt", "B", "C"):
            setattr(piece, name, getattr(prob, name)[lo:hi])
        o, conv, h = run_gpu_prefill(piece, flags, 4096, conv, h)
        outs.append(o)
    assert np.array_equal(np.concatenate(outs), whole[0]) and np.array_equal(conv, whole[1]) and np.array_equal(h, whole[2])


def _tree_rig(regime, act, powers, g, Dn=200):
    cfg = parity.small_config(Dn, act, cid=93)
    rig = TreeRig(cfg, gen.paper_tree((3, 2, 2, 1, 1)), conv_bias=True, general_A=not powers)
    shape_A(rig.params, regime, powers, g)
    rig.dt, raw = shape_dt(rig.dt, rig.params, regime, act, g)
    rig.flags = flags_for(raw, powers)
    rig.lay = upload_layer(rig.params, act, rig.flags)
    rig.dev = [to_device(a, rig.tdt) for a in (rig.x, rig.z, rig.dt, rig.B, rig.C)]
    return rig


@pytest.mark.parametrize("regime", REGIMES)
@pytest.mark.parametrize("act", ["f32", "bf16"])
@pytest.mark.parametrize("powers", [False, True])
def test_tree_step_outside_the_recipe(regime, act, powers):
    g = np.random.default_rng(case_seed(regime, act, powers, 1))
    rig = _tree_rig(regime, act, powers, g)
    out = rig.run_levels()
    assert int(rig.status.item()) == 0
    o_out, o_conv, o_h = rig.oracle()
    assert_close(out.float().cpu().numpy(), o_out, TOL[act], "node outputs")
    h, conv = rig.states()
    assert_close(h, o_h, TOL_STATE, "node SSM states")
    assert np.array_equal(conv.astype(np.float64), o_conv)


@pytest.mark.parametrize("act", ["f32", "bf16"])
@pytest.mark.parametrize("powers", [False, True])
def test_tree_step_with_zero_step_size_copies_the_parent_state_bit_for_bit(act, powers):
    g = np.random.default_rng(23)
    rig = _tree_rig("", act, powers, g)
    rig.dt = np.zeros_like(rig.dt)
    rig.params.dt_bias[:] = 0.0
    rig.flags = flags_for(True, powers)
    rig.lay = upload_layer(rig.params, act, rig.flags)
    rig.dev = [to_device(a, rig.tdt) for a in (rig.x, rig.z, rig.dt, rig.B, rig.C)]
    out = rig.run_levels()
    assert int(rig.status.item()) == 0
    h, _ = rig.states()
    for i in range(rig.tree.n_nodes):
        assert np.array_equal(h[i].view(np.uint32), rig.h0.view(np.uint32)), f"node {i}: every state of the tree is the committed state"
    o_out, _, _ = rig.oracle()
    assert_close(out.float().cpu().numpy(), o_out, TOL[act], "node outputs")


@pytest.mark.parametrize("regime", REGIMES)
@pytest.mark.parametrize("act", ["f32", "bf16"])
@pytest.mark.parametrize("powers", [False, True])
def test_projection_step_outside_the_recipe(regime, act, powers):
    """The same regimes through the step that forms dt, B and C itself: the step size is shaped through W_dt and
    the bias (large spread for big_dt; non-negative weights times a non-negative input are not available, so
    zero_dt uses W_dt = 0 with a bias that is 0 on half of the channels and small on the others)."""
    g = np.random.default_rng(case_seed(regime, act, powers, 2))
    Dn, R = 392, 16
    cfg = parity.small_config(Dn, act, cid=93)
    rig = ProjRig(cfg, gen.paper_tree((3, 3, 2, 1)), R, conv_bias=True, general_A=not powers)
    shape_A(rig.params, regime, powers, g)
    raw = False
    if regime == "big_dt":
        rig.W_dt = gen.round_to_act(rig.W_dt * np.float32(40.0), act)   # projected pre-activations of spread ~20
    elif regime == "zero_dt":
        raw = True
        rig.W_dt = np.zeros_like(rig.W_dt)
        rig.params.dt_bias[:] = np.where(np.arange(Dn) % 2 == 0, 0.0, g.uniform(0.001, 0.2, size=Dn)).astype(np.float32)
    rig.flags = flags_for(raw, powers)
    rig.lay = upload_layer(rig.params, act, rig.flags)
    rig.dW_dt = to_device(rig.W_dt, rig.tdt)
    out = rig.run_levels()
    assert int(rig.status.item()) == 0
    o_out, o_conv, o_h, _, _, _ = rig.oracle()
    assert_close(out.float().cpu().numpy(), o_out, TOL[act], "node outputs")
    h, conv = rig.states()
    assert_close(h, o_h, TOL_STATE, "node SSM states")
    assert np.array_equal(conv.astype(np.float64), o_conv)
    if regime == "zero_dt":   # channels whose step size is exactly 0 keep the committed state in every node
        even = np.arange(Dn) % 2 == 0
        for i in range(rig.tree.n_nodes):
            assert np.array_equal(h[i][even].view(np.uint32), rig.h0[even].view(np.uint32))
