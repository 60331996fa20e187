"""Calls over several layers (one launch for all of them) against one call per layer, and the prefill's plans against each other:
unsplit blocks of 128 and 256 channels, sequences handed out longest first, a workspace that only fewer chunks fit."""

import numpy as np
import pytest
import torch

import gen
import oracle
import parity
from parity import TOL, TOL_STATE, assert_close

pytestmark = pytest.mark.gpu

import paper_2506_01206_b200 as md
from paper_2506_01206_b200.device_inputs import i32, to_device, torch_act, upload_layer
from paper_2506_01206_b200.stack import DrafterStack


def _problems(n_layers, Dn, act, lens, general_A):
    return [parity.make_problem(parity.small_config(Dn, act, len(lens), cid=60 + l), lens, conv_bias=True, general_A=general_A) for l in range(n_layers)], torch_act(act)


@pytest.mark.parametrize("n_layers,Dn,act,lens,general_A", [
    (2, 64, "f32", [1], False), (3, 200, "bf16", [70, 0, 5, 33], True), (33, 136, "bf16", [40], False), (24, 1536, "bf16", [150], False),
    (2, 264, "f32", [300, 17], True), (5, 384, "bf16", [3, 90, 89, 90, 1], False)])
def test_stack_prefill_matches_oracle(n_layers, Dn, act, lens, general_A):
    probs, tdt = _problems(n_layers, Dn, act, lens, general_A)
    flags = md.MDRAFT_DT_SOFTPLUS | (0 if general_A else md.MDRAFT_A_POWERS)
    T, S = sum(lens), len(lens)
    stack = DrafterStack([upload_layer(p.params, act, flags) for p in probs], S, T, S, max(lens))
    ins = [tuple(to_device(a, tdt) for a in (p.x, p.z, p.dt, p.B, p.C)) for p in probs]
    outs = list(torch.full((n_layers, T, Dn), float("nan"), dtype=tdt, device="cuda"))
    stack.prefill(ins, outs, i32(probs[0].cu), max(lens), None, i32(np.arange(S)))
    torch.cuda.synchronize()
    stack.check_status()
    for l in {0, n_layers // 2, n_layers - 1}:
        p = probs[l]
        o_out, o_conv, o_h = oracle.prefill(oracle.layer_from_params(p.params), p.x, p.z, p.dt, p.B, p.C, p.cu)
        assert_close(outs[l].float().cpu().numpy(), o_out, TOL[act], f"out of layer {l}")
        assert_close(stack.cache.ssm[l].cpu().numpy(), o_h, TOL_STATE, f"state of layer {l}")
        assert np.array_equal(stack.cache.conv[l].float().cpu().numpy().astype(np.float64), o_conv)


@pytest.mark.parametrize("act", ["f32", "bf16"])
def test_stack_prefill_of_a_general_A_in_three_kernels_matches_oracle(act):
    """Too much work for the one-kernel form: the summary pass, the carry scan and the output pass over several layers."""
    n_layers, Dn, lens = 3, 520, [1500, 0, 700]
    probs, tdt = _problems(n_layers, Dn, act, lens, True)
    lays = [upload_layer(p.params, act, md.MDRAFT_DT_SOFTPLUS) for p in probs]
    T, S = sum(lens), len(lens)
    assert md.mdraft_prefill_stack_launches(lays[0], n_layers, T, S, max(lens)) == 3
    stack = DrafterStack(lays, 2 * S, T, S, max(lens))
    g = np.random.default_rng(8)
    h0 = g.normal(size=(n_layers, S, Dn, 16)).astype(np.float32)
    c0 = gen.round_to_act(g.normal(size=(n_layers, S, 3, Dn)).astype(np.float32), act)
    stack.cache.ssm[:, S:], stack.cache.conv[:, S:] = torch.from_numpy(h0).cuda(), to_device(c0, tdt)
    ins = [tuple(to_device(a, tdt) for a in (p.x, p.z, p.dt, p.B, p.C)) for p in probs]
    outs = list(torch.full((n_layers, T, Dn), float("nan"), dtype=tdt, device="cuda"))
    assert md.mdraft_conv_scan_prefill_stack(lays, range(n_layers), stack.cache, ins, outs, i32(probs[0].cu), max(lens), i32(np.arange(S, 2 * S)), i32(np.arange(S)),
                                             stack.workspace, stack.status)
    torch.cuda.synchronize()
    stack.check_status()
    for l, p in enumerate(probs):
        o_out, o_conv, o_h = oracle.prefill(oracle.layer_from_params(p.params), p.x, p.z, p.dt, p.B, p.C, p.cu, c0[l], h0[l])
        assert_close(outs[l].float().cpu().numpy(), o_out, TOL[act], f"out of layer {l}")
        assert_close(stack.cache.ssm[l, :S].cpu().numpy(), o_h, TOL_STATE, f"state of layer {l}")
        assert np.array_equal(stack.cache.conv[l, :S].float().cpu().numpy().astype(np.float64), o_conv)


def test_layers_whose_tensors_overlap_run_in_order():
    probs, tdt = _problems(3, 64, "f32", [50], False)
    layers = [upload_layer(p.params, "f32") for p in probs]
    x, z, dt, B, C = (to_device(a, tdt) for a in (probs[0].x, probs[0].z, probs[0].dt, probs[0].B, probs[0].C))
    a, b = torch.empty((50, 64), device="cuda"), torch.empty((50, 64), device="cuda")
    one, chain = DrafterStack(layers, 1, 50, 1, 50), DrafterStack(layers, 1, 50, 1, 50)
    ins, outs = [(x, z, dt, B, C), (a, z, dt, B, C), (b, z, dt, B, C)], [a, b, a]   # layer l + 1 reads what layer l writes
    assert not md.mdraft_conv_scan_prefill_stack(layers, range(3), chain.cache, ins, outs, None, 50, None, i32([0]), chain.workspace, chain.status)
    chain.prefill(ins, outs, None, 50, None, i32([0]))
    got = a.clone()
    for l in range(3):
        one.prefill(ins, outs, None, 50, None, i32([0]), layer_range=[l])
    torch.cuda.synchronize()
    assert torch.equal(got, a) and torch.equal(one.cache.ssm, chain.cache.ssm)


@pytest.mark.parametrize("n_layers", [2, 33])
def test_stack_tree_round_equals_layer_by_layer(n_layers):
    probs, tdt = _problems(n_layers, 136, "bf16", [12], False)
    layers = [upload_layer(p.params, "bf16") for p in probs]
    ins = [tuple(to_device(a, tdt) for a in (p.x, p.z, p.dt, p.B, p.C)) for p in probs]
    parent, node, levels = i32([0, 1, 1, 1, 2, 2, 3, 4, 5, 5, 6, 7]), i32(np.arange(1, 13)), [0, 1, 4, 4, 8, 12]
    res = []
    for ranges in ([range(n_layers)], [[l] for l in range(n_layers)]):
        st = DrafterStack(layers, 13, 1, 1, 1)
        st.cache.ssm[:, 0] = torch.randn((n_layers, 136, 16), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
        outs = list(torch.empty((n_layers, 12, 136), dtype=tdt, device="cuda"))
        for r in ranges:
            st.tree_round(ins, outs, parent, node, levels, layer_range=r)
        torch.cuda.synchronize()
        st.check_status()
        res.append((torch.stack(outs), st.cache.ssm, st.cache.conv))
    for a, b in zip(*res):
        assert torch.equal(a, b)


def test_a_workspace_for_fewer_chunks_still_serves():
    Dn, lens = 152, [30000, 10000]
    prob = parity.make_problem(parity.small_config(Dn, "bf16", 2), lens)
    lay, dev = upload_layer(prob.params, "bf16"), [to_device(a, torch.bfloat16) for a in (prob.x, prob.z, prob.dt, prob.B, prob.C)]
    need = md.mdraft_prefill_workspace_bytes(lay, 40000, 2, 30000)
    res = []
    for n in (need, need * 3 // 4):
        cache, out = md.StateCache(1, 2, Dn), torch.empty((40000, Dn), dtype=torch.bfloat16, device="cuda")
        md.mdraft_conv_scan_prefill(lay, cache, 0, *dev, out, i32(prob.cu), 30000, None, i32([0, 1]), torch.empty(n, dtype=torch.uint8, device="cuda"))
        torch.cuda.synchronize()
        res.append((out.float(), cache.ssm))
    assert_close(res[1][0].cpu().numpy(), res[0][0].cpu().numpy().astype(np.float64), TOL["bf16"], "out")
    assert_close(res[1][1].cpu().numpy(), res[0][1].cpu().numpy().astype(np.float64), TOL_STATE, "state")
    with pytest.raises(md.MdraftError):
        md.mdraft_conv_scan_prefill(lay, cache, 0, *dev, out, i32(prob.cu), 30000, None, i32([0, 1]), torch.empty(256, dtype=torch.uint8, device="cuda"))
