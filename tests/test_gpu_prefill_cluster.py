"""The one-kernel form of the context encode (the chunks of a sequence are the warps of a thread-block cluster), where the default
plan takes it: against the fp64 oracle, and against the three-kernel form of the same call.

Tolerances: those of the other encodes (tests/parity.py).  The two forms differ by where they cut a sequence, and across a cut a state
decays by the exponential of the summed step sizes instead of a product of one per token.  A token's factor for A = -n is good to n 2^-22
(powers of one approximate exponential, whose error has the same sign in all of them) and some 1 / (n Delta) = 100 / n tokens count, so the two
may be 100 * 2^-22 = 2.4e-5 apart; the largest of some 10^5 elements, taken relative to its value or the RMS, lies up to four times that
out: 1e-4.  bf16 outputs are besides rounded once each, 2^-8 of the value at most apart when a tie falls, with the RMS floor 2^-7."""

import ctypes

import numpy as np
import pytest
import torch

import parity
from parity import TOL, TOL_STATE, assert_close
from test_gpu_parity_small import random_state, run_gpu_prefill, run_oracle_prefill

pytestmark = pytest.mark.gpu

import paper_2506_01206_b200 as md
from paper_2506_01206_b200.device_inputs import i32, to_device, torch_act, upload_layer

TOL_FORMS = 1e-4

# act, D, lengths, (blocks, warps) that the rule gives with A = powers and with a general A; (0, 0): so short that the output pass alone is as fast
SHAPES = [
    ("f32", 8, [1], (0, 0), (0, 0)), ("bf16", 8, [3], (0, 0), (0, 0)), ("bf16", 1496, [31, 32, 33], (0, 0), (0, 0)),
    ("bf16", 32, [64], (4, 4), (4, 4)), ("f32", 64, [256], (8, 8), (8, 8)), ("bf16", 40, [65, 1, 0, 4, 257], (6, 4), (6, 4)),
    ("f32", 200, [33, 500], (6, 8), (6, 8)), ("bf16", 768, [256], (4, 8), (4, 8)), ("bf16", 1536, [130], (5, 4), (5, 4)),
    ("f32", 1000, [17, 90], (3, 8), (3, 8)), ("bf16", 72, [511], (8, 8), (8, 8)), ("f32", 24, [2, 0, 1, 500], (8, 8), (8, 8)),
    ("bf16", 768, [64, 63, 1, 4], (1, 8), (1, 8)), ("f32", 768, [48, 3, 0, 47], (1, 4), (3, 4)), ("bf16", 768, [64, 2], (2, 8), (2, 8)),
    ("f32", 136, [32, 32], (1, 8), (2, 4)), ("f32", 520, [300, 299], (7, 4), (7, 4))]


def form(layer, n_layers, lens, shared=False):
    """(blocks, warps) of the one-kernel form that a call takes, (0, 0) for the plan's own kernels; shared: several sequences that would be cut have
    both starting and final slots."""
    f = md.load_library().mdraft_internal_prefill_form(ctypes.byref(layer.c()), n_layers, sum(lens), len(lens), max(lens), int(shared))
    return f // 256, f % 256


@pytest.mark.parametrize("act,Dn,lens,powers_form,general_form", SHAPES)
@pytest.mark.parametrize("general_A", [False, True])
def test_one_kernel_form_matches_oracle_and_the_general_form(act, Dn, lens, powers_form, general_form, general_A):
    cfg = parity.small_config(Dn, act, len(lens), cid=97)
    prob = parity.make_problem(cfg, lens, conv_bias=True, general_A=general_A)
    flags = md.MDRAFT_DT_SOFTPLUS | (0 if general_A else md.MDRAFT_A_POWERS)
    lay = upload_layer(prob.params, act, flags)
    assert form(lay, 1, lens) == (general_form if general_A else powers_form)
    ci, hi = random_state(cfg, len(lens), 7)
    for init, strided, in_place in ((False, False, False), (True, True, False), (True, False, True)):
        state = (ci, hi) if init else (None, None)
        got = run_gpu_prefill(prob, flags, 0, *state, in_place=in_place, strided=strided)
        o_out, o_conv, o_h = run_oracle_prefill(prob, flags, *state)
        assert_close(got[0], o_out, TOL[act], "out")
        assert_close(got[2], o_h, TOL_STATE, "final SSM state")
        assert np.array_equal(got[1], o_conv)
        other = run_gpu_prefill(prob, flags, 32, *state, in_place=in_place, strided=strided)
        assert_close(got[0], other[0], TOL_FORMS if act == "f32" else 2 ** -7, "out, other form")
        assert_close(got[2], other[2], TOL_FORMS, "state, other form")
        assert np.array_equal(got[1], other[1])


@pytest.mark.parametrize("act", ["f32", "bf16"])
def test_one_kernel_form_of_a_stack_and_its_faults(act):
    """Several layers in one launch; a sequence with a slot out of range and one with malformed offsets are left out alone."""
    lens, Dn, NL = [50, 70, 20], 136, 3
    tdt = torch_act(act)
    probs = [parity.make_problem(parity.small_config(Dn, act, 3, cid=70 + l), lens) for l in range(NL)]
    flags = md.MDRAFT_DT_SOFTPLUS | md.MDRAFT_A_POWERS
    lays = [upload_layer(p.params, act, flags) for p in probs]
    assert form(lays[0], NL, lens) == (5, 4)
    cache = md.StateCache(NL, 3, Dn, act=tdt)
    cache.ssm.fill_(5.0)
    out = torch.full((NL, sum(lens), Dn), 9.0, dtype=tdt, device="cuda")
    ins = [tuple(to_device(a, tdt) for a in (p.x, p.z, p.dt, p.B, p.C)) for p in probs]
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(max(256, md.mdraft_prefill_stack_workspace_bytes(lays[0], NL, sum(lens), 3, max(lens))), dtype=torch.uint8, device="cuda")
    assert md.mdraft_conv_scan_prefill_stack(lays, range(NL), cache, ins, list(out), i32([0, 50, 120, 140]), max(lens), None, i32([0, 7, 2]), ws, status)
    torch.cuda.synchronize()
    assert int(status.item()) == md.MDRAFT_DEV_BAD_SLOT
    assert bool((out[:, 50:120] == 9.0).all()) and bool((cache.ssm[:, 1] == 5.0).all())
    for l, p in enumerate(probs):
        o_out, _, o_h = run_oracle_prefill(p, flags)
        for s, (a, b) in ((0, (0, 50)), (2, (120, 140))):
            assert_close(out[l, a:b].float().cpu().numpy(), o_out[a:b], TOL[act], f"layer {l} sequence {s}")
            assert_close(cache.ssm[l, s].cpu().numpy(), o_h[s], TOL_STATE, f"layer {l} state {s}")
    status.zero_(); out.fill_(9.0)
    assert md.mdraft_conv_scan_prefill_stack(lays, range(NL), cache, ins, list(out), i32([0, 50, 200, 140]), max(lens), None, i32([0, 1, 2]), ws, status)
    torch.cuda.synchronize()
    assert int(status.item()) == md.MDRAFT_DEV_BAD_SEQLENS
    assert not bool((out[:, :50] == 9.0).all()) and bool((out[:, 50:] == 9.0).all())


@pytest.mark.parametrize("act,Dn,n_layers,lens,in_one", [
    ("bf16", 200, 1, [150, 0, 140, 1, 90], True), ("f32", 72, 2, [400, 333, 0, 500], True), ("bf16", 520, 2, [900, 850, 700], False)])
def test_sequences_may_start_from_a_slot_that_one_of_them_stores_to(act, Dn, n_layers, lens, in_one):
    """Several sequences continue from one prefix's slot and the first stores its state back there: all of them start from what the slot
    held before the call, bit for bit as from a slot that nobody stores to.  (The one-kernel form delivers the final states by a second kernel then.)"""
    S, T, tdt = len(lens), sum(lens), torch_act(act)
    probs = [parity.make_problem(parity.small_config(Dn, act, S, cid=60 + l), lens) for l in range(n_layers)]
    flags = md.MDRAFT_DT_SOFTPLUS | md.MDRAFT_A_POWERS
    lays = [upload_layer(p.params, act, flags) for p in probs]
    assert (form(lays[0], n_layers, lens, shared=True) != (0, 0)) == in_one
    ci, hi = random_state(probs[0].cfg, 1, 7)
    ins = [tuple(to_device(a, tdt) for a in (p.x, p.z, p.dt, p.B, p.C)) for p in probs]
    ws = torch.empty(md.mdraft_prefill_stack_workspace_bytes(lays[0], n_layers, T, S, max(lens)), dtype=torch.uint8, device="cuda")
    res = []
    for start in (0, S):
        cache = md.StateCache(n_layers, S + 1, Dn, act=tdt)
        cache.ssm.fill_(float("nan")); cache.conv.fill_(float("nan"))
        cache.ssm[:, start], cache.conv[:, start] = torch.from_numpy(np.asarray(hi[0], dtype=np.float32)).cuda(), to_device(ci[0], tdt)
        outs = list(torch.full((n_layers, T, Dn), float("nan"), dtype=tdt, device="cuda"))
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        if n_layers == 1:
            md.mdraft_conv_scan_prefill(lays[0], cache, 0, *ins[0], outs[0], i32(probs[0].cu), max(lens), i32([start] * S), i32(np.arange(S)), ws, 0, status)
        else:
            assert md.mdraft_conv_scan_prefill_stack(lays, range(n_layers), cache, ins, outs, i32(probs[0].cu), max(lens), i32([start] * S), i32(np.arange(S)), ws, status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        res.append((torch.stack(outs), cache.ssm[:, :S], cache.conv[:, :S]))
    for a, b in zip(*res):
        assert torch.equal(a, b)
    for l, p in enumerate(probs):
        o_out, o_conv, o_h = run_oracle_prefill(p, flags, np.repeat(ci[:1], S, 0), np.repeat(hi[:1], S, 0))
        assert_close(res[0][0][l].float().cpu().numpy(), o_out, TOL[act], f"out of layer {l}")
        assert_close(res[0][1][l].cpu().numpy(), o_h, TOL_STATE, f"states of layer {l}")
        assert np.array_equal(res[0][2][l].float().cpu().numpy().astype(np.float64), o_conv)


@pytest.mark.parametrize("act", ["f32", "bf16"])
@pytest.mark.parametrize("general_A", [False, True])
def test_an_infinite_A_forgets_and_nothing_else(act, general_A):
    """-exp(A_log) of a large A_log is -inf: such a state is its last input alone.  In every form, also where a chunk's decay is formed from a sum of
    step sizes (inf times the 0 of a sequence's first chunk is not a number)."""
    Dn, lens = 136, [256]
    prob = parity.make_problem(parity.small_config(Dn, act, 1, cid=97), lens, general_A=general_A)
    prob.params.A[::3] = -np.inf
    if general_A:
        prob.params.A[1::3, 5] = -np.inf
    flags = md.MDRAFT_DT_SOFTPLUS | (0 if general_A else md.MDRAFT_A_POWERS)
    assert form(upload_layer(prob.params, act, flags), 1, lens) != (0, 0)
    state = random_state(prob.cfg, 1, 7)
    o_out, o_conv, o_h = run_oracle_prefill(prob, flags, *state)
    for chunk_len in (0, 32, 4096):
        got = run_gpu_prefill(prob, flags, chunk_len, *state)
        assert_close(got[0], o_out, TOL[act], f"out, chunk_len {chunk_len}")
        assert_close(got[2], o_h, TOL_STATE, f"final SSM state, chunk_len {chunk_len}")
        assert np.array_equal(got[1], o_conv)
