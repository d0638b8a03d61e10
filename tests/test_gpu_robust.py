"""GPU results on scenes as training leaves them at their worst: Gaussians whose
values are not finite (they must count for nothing, and change nothing of the
others') and centres far from all others."""
import numpy as np
import pytest
import torch

from paper_2410_14462_gb300 import inputs, ludvig
from tests.gpu_util import device_features, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2410_14462_gb300 import build
    build.build()
    ludvig.load()


def _with_opacity(scene, idx, value):
    op = scene.opacity.copy()
    op[idx] = value
    return inputs.Scene(scene.means, scene.scales, scene.quats, op)


# 5 views of 30 x 17 tiles (2550 items) are above, and one view is below, the
# limits of the few-tile kernels.  A NaN fails alpha >= 1/255, so the Gaussian is
# skipped like one of opacity 0; sums of float32 in another order: 1e-5.
@pytest.mark.parametrize("views", [5, 1])
@pytest.mark.parametrize("d,dtype", [(1, torch.float32), (3, torch.bfloat16), (40, torch.float32), (40, torch.bfloat16),
                                     (33, torch.float32)])
def test_opacity_not_a_number_has_no_weight(d, dtype, views):
    wl = inputs.small_field_workload(n=6000, views=views, d=d, width=475, height=269)
    bad = np.arange(0, 6000, 97)
    F = device_features(wl, range(views), dtype=dtype)
    ref, bref = ludvig.uplift(ludvig.Scene.from_inputs(_with_opacity(wl.scene, bad, 0.0)), wl.cams.params, 475, 269, F)
    got, beta = ludvig.uplift(ludvig.Scene.from_inputs(_with_opacity(wl.scene, bad, np.nan)), wl.cams.params, 475, 269, F)
    assert (got[bad] == 0).all() and (beta[bad] == 0).all()
    assert torch.isfinite(got).all() and (bref > 0).sum() > 1000
    assert rel_l2(beta.cpu().numpy(), bref.cpu().numpy()) <= 1e-5
    assert rel_l2(got.cpu().numpy(), ref.cpu().numpy()) <= 1e-5


def test_opacity_not_a_number_is_not_rendered():
    wl = inputs.small_field_workload(n=6000, views=5, d=40, width=475, height=269)
    bad = np.arange(0, 6000, 97)
    f = torch.randn((6000, 40), device="cuda", generator=torch.Generator("cuda").manual_seed(0))
    ref, got = (ludvig.render(ludvig.Scene.from_inputs(_with_opacity(wl.scene, bad, v)), wl.cams.params, 475, 269, f)
                for v in (0.0, np.nan))
    assert rel_l2(got.cpu().numpy(), ref.cpu().numpy()) <= 1e-5
