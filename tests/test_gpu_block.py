"""One generation of the block stack in its own kernels (mdraft_block_generation) against the fp64 replica of the drafter
tests: row tiles of 32, column tiles of 16 and 32 with ragged last ones, contractions that leave warps without work, that take
every warp round its loop a second time, and the longest ones supported.

Tolerance: xz, y and h of each of the two layers and the logits are rounded to bf16, seven roundings of 2^-9 / sqrt(3) of the value in the
root mean square; together 3e-3 of a logit's RMS, and the largest of some 10^5 logits lies five times that out: 1.5e-2."""

import pytest
import torch

from parity import assert_close
from test_gpu_drafter import _replica_logits

pytestmark = pytest.mark.gpu

import paper_2506_01206_b200 as md
from paper_2506_01206_b200.drafter import ToyDrafter


TOL_LOGITS = 2e-2


def _drafter(width, d_model, d_inner, vocab):
    """A two-layer stack with a committed state, and that state in fp64."""
    d = ToyDrafter(n_layers=2, d_model=d_model, d_inner=d_inner, dt_rank=8, vocab=vocab, max_nodes=width, seed=width)
    assert d.block_kernels
    g = torch.Generator(device="cuda").manual_seed(2)
    d.cache.ssm[:, 0] = torch.randn(d.cache.ssm[:, 0].shape, generator=g, device="cuda")
    d.cache.conv[:, 0] = torch.randn(d.cache.conv[:, 0].shape, generator=g, device="cuda")
    return d, g, d.cache.conv[:, 0].double().cpu().numpy(), d.cache.ssm[:, 0].double().cpu().numpy()


@pytest.mark.parametrize("width,d_model,d_inner,vocab", [
    (1, 32, 64, 96), (8, 96, 96, 104), (17, 64, 128, 1192), (32, 64, 640, 3600), (33, 256, 64, 88), (64, 288, 160, 9800), (5, 1056, 64, 4000),
    (33, 416, 1216, 96),     # two row tiles, in_proj in tiles of 32 columns: both loops without fragments ahead, a second time round
    (64, 416, 64, 2376),     # two row tiles, in_proj in tiles of 16 columns over more than twelve blocks of the contraction
    (3, 64, 1568, 96), (32, 1408, 2048, 4736),   # out_proj beyond the fragments held ahead of the wait; the largest shapes supported
    (9, 800, 64, 4744)])     # the longest contraction of the persistent form
def test_generation_matches_path_replica(width, d_model, d_inner, vocab):
    d, g, conv0, h0 = _drafter(width, d_model, d_inner, vocab)
    d.tokens.copy_(torch.randint(0, vocab, (width,), generator=g, device="cuda"))
    d.node_slot.copy_(torch.arange(1, width + 1, device="cuda"))
    d.logits.fill_(float("nan"))
    for use_graph in (False, True):
        d.generation(0, width, use_graph=use_graph)
        torch.cuda.synchronize()
        assert int(d.status.item()) == 0
        logits, toks = d.logits.double().cpu().numpy(), d.tokens.cpu().numpy()
        for v in {0, width // 2, width - 1}:
            assert_close(logits[v], _replica_logits(d, [int(toks[v])], conv0, h0), TOL_LOGITS, f"node {v}")


@pytest.mark.parametrize("up,width,d_model,d_inner", [(1, 1, 64, 64), (5, 18, 96, 160), (20, 40, 416, 1216)])
def test_a_generation_below_a_generation_matches_path_replica(up, width, d_model, d_inner):
    """Nodes whose parents are nodes: states and windows come from, and go to, slots that a generation wrote."""
    vocab = 104
    d, g, conv0, h0 = _drafter(up + width, d_model, d_inner, vocab)
    d.tokens.copy_(torch.randint(0, vocab, (up + width,), generator=g, device="cuda"))
    d.node_slot.copy_(torch.arange(1, up + width + 1, device="cuda"))
    parent = [7 * j % up for j in range(width)]
    d.parent_slot.copy_(torch.tensor([0] * up + [1 + p for p in parent]))
    d.generation(0, up)
    d.generation(up, up + width)
    torch.cuda.synchronize()
    assert int(d.status.item()) == 0
    logits, toks = d.logits.double().cpu().numpy(), d.tokens.cpu().numpy()
    for j in {0, width // 2, width - 1}:
        want = _replica_logits(d, [int(toks[parent[j]]), int(toks[up + j])], conv0, h0)
        assert_close(logits[up + j], want, TOL_LOGITS, f"node {up + j}")


def test_a_token_outside_the_vocabulary_is_flagged():
    d = ToyDrafter(n_layers=1, d_model=32, d_inner=64, dt_rank=8, vocab=96, max_nodes=2)
    d.tokens.copy_(torch.tensor([3, 96]))
    d.node_slot.copy_(torch.tensor([1, 2]))
    d.generation(0, 2, use_graph=False)
    torch.cuda.synchronize()
    assert int(d.status.item()) == md.MDRAFT_DEV_BAD_SLOT
    assert bool(torch.isfinite(d.logits[0].float()).all()) and float(d.logits[1].float().abs().max()) == 0.0
