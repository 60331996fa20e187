"""One generation of the block stack in its own kernels (mdraft_block_generation) against the fp64 replica of the drafter
tests: row tiles of 32, column tiles of 8, 24 and 32 with ragged last ones, contractions that leave warps without work."""

import pytest
import torch

from parity import assert_close
from test_gpu_drafter import _replica_logits

pytestmark = pytest.mark.gpu

import paper_2506_01206_b200 as md
from paper_2506_01206_b200.drafter import ToyDrafter


@pytest.mark.parametrize("width,d_model,d_inner,vocab", [
    (1, 32, 64, 96), (8, 96, 96, 104), (17, 64, 128, 1192), (32, 64, 640, 3600), (33, 256, 64, 88), (64, 288, 160, 9800), (5, 1056, 64, 4000)])
def test_generation_matches_path_replica(width, d_model, d_inner, vocab):
    d = ToyDrafter(n_layers=2, d_model=d_model, d_inner=d_inner, dt_rank=8, vocab=vocab, max_nodes=width, seed=width)
    assert d.block_kernels
    g = torch.Generator(device="cuda").manual_seed(2)
    d.cache.ssm[:, 0] = torch.randn(d.cache.ssm[:, 0].shape, generator=g, device="cuda")
    d.cache.conv[:, 0] = torch.randn(d.cache.conv[:, 0].shape, generator=g, device="cuda")
    conv0, h0 = d.cache.conv[:, 0].double().cpu().numpy(), d.cache.ssm[:, 0].double().cpu().numpy()
    d.tokens.copy_(torch.randint(0, vocab, (width,), generator=g, device="cuda"))
    d.node_slot.copy_(torch.arange(1, width + 1, device="cuda"))
    d.logits.fill_(float("nan"))
    for use_graph in (False, True):
        d.generation(0, width, use_graph=use_graph)
        torch.cuda.synchronize()
        assert int(d.status.item()) == 0
        logits, toks = d.logits.double().cpu().numpy(), d.tokens.cpu().numpy()
        for v in {0, width // 2, width - 1}:
            assert_close(logits[v], _replica_logits(d, [int(toks[v])], conv0, h0), 3e-2, f"node {v}")


def test_a_token_outside_the_vocabulary_is_flagged():
    d = ToyDrafter(n_layers=1, d_model=32, d_inner=64, dt_rank=8, vocab=96, max_nodes=2)
    d.tokens.copy_(torch.tensor([3, 96]))
    d.node_slot.copy_(torch.tensor([1, 2]))
    d.generation(0, 2, use_graph=False)
    torch.cuda.synchronize()
    assert int(d.status.item()) == md.MDRAFT_DEV_BAD_SLOT
    assert bool(torch.isfinite(d.logits[0].float()).all()) and float(d.logits[1].float().abs().max()) == 0.0
