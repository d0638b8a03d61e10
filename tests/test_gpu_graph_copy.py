"""Diffusion of several columns and reachability run on the CSR for a few steps and on a
renumbered copy of it from then on: the same results on either, and the present
values' after a change.  One diffusion step sums the same products in the same order on
both, scaled by norms summed in another order: 1e-6 relative L2; reachability is exact."""
import numpy as np
import pytest
import torch

from paper_2410_14462_gb300 import inputs, ludvig
from tests.gpu_util import rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2410_14462_gb300 import build
    build.build()
    ludvig.load()


def _graph(n=6000, k=8):
    s = inputs.scene_clusters(n, seed=9, n_clusters=5, sigma=0.1, extent=1.0)
    f = torch.randn((n, 24), device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    g = ludvig.Graph.rbf(ludvig.Scene.from_inputs(s), k, f)
    g.reweight(0.5, None, binarize=0.0, row_normalize=True)
    return g


@pytest.mark.parametrize("dx", [2, 5, 32])
def test_few_and_many_diffusion_steps(dx):
    g = _graph()
    x = torch.rand((6000, dx), device="cuda", generator=torch.Generator("cuda").manual_seed(dx))
    before = g.workspace_bytes()
    one, two = g.diffuse(x, 1), g.diffuse(x, 2)
    copied = _graph()
    copied.diffuse(x, 50)   # makes the copy
    assert rel_l2(copied.diffuse(x, 1).cpu().numpy(), one.cpu().numpy()) <= 1e-6
    assert rel_l2(copied.diffuse(x, 2).cpu().numpy(), two.cpu().numpy()) <= 1e-6
    assert before < g.workspace_bytes() < copied.workspace_bytes()   # three steps in all: no copy yet
    again = g.diffuse(x, 1)                                          # the fourth
    assert g.workspace_bytes() >= copied.workspace_bytes() * 0.9
    assert rel_l2(again.cpu().numpy(), one.cpu().numpy()) <= 1e-6


def test_reach_on_either_and_after_a_change():
    x = torch.zeros((6000, 3), device="cuda")
    x[5, 0] = x[100, 1] = x[4000, 2] = 1.0
    few, many = _graph(), _graph()
    many.reach_weight(x, 40)
    for steps in (1, 7):
        assert torch.equal(few.reach_weight(x, steps), many.reach_weight(x, steps))
    unary = torch.rand((6000,), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    for g in (few, many):   # other values, of which many are zero
        g.reweight(0.05, unary, binarize=0.2, row_normalize=False)
    fresh = _graph()
    fresh.reweight(0.05, unary, binarize=0.2, row_normalize=False)
    ref = fresh.reach_weight(x, 20)
    assert torch.equal(few.reach_weight(x, 20), ref) and torch.equal(many.reach_weight(x, 20), ref)
    assert torch.equal(fresh.reach_weight(x, 20), ref)   # by then on the copy
    y = torch.rand((6000, 2), device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    assert rel_l2(many.diffuse(y, 1).cpu().numpy(), fresh.diffuse(y, 1).cpu().numpy()) <= 1e-6
