"""GPU parity at the sizes where the kernels' splits can go wrong: launches with
more tiles than the few-tile kernels take, widths the tensor cores do not take
(whole and ragged channel blocks, several of them), features that are not
finite, views that end inside or off a quantiser piece, and the graph kernels'
width and column remainders.  Bars: float32 uplift 1e-5 relative L2 against the
float64 oracle, bfloat16 1e-2, weights and one diffusion step 1e-5, codes,
scales and neighbours bit-exact."""
import numpy as np
import pytest
import torch

import oracle
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


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("elems", [1, 4096, 8192 + 5, 16384])
def test_quantize_pieces(dtype, elems):
    x = np.random.default_rng(elems).normal(size=(3, elems)).astype(np.float32)
    xt = torch.from_numpy(x).to(dtype).cuda()
    q, s = ludvig.fp8_quantize(xt)
    qr, sr = oracle.fp8_quantize(xt.float().cpu().numpy())
    assert np.array_equal(s.cpu().numpy(), sr) and np.array_equal(q.cpu().numpy(), qr)


@pytest.mark.parametrize("n,d,nq,k", [(1, 1, 1, 1), (31, 13, 3, 1), (33, 48, 5, 3), (20_011, 100, 11, 4),
                                      (4097, 512, 21, 4), (300, 640, 60, 4), (2000, 5120, 4, 4)])
def test_relevancy_sizes(n, d, nq, k):
    rng = np.random.default_rng(n + d)
    f, pq, pc = (rng.normal(size=(m, d)).astype(np.float32) for m in (n, nq, k))
    got = ludvig.relevancy(*(torch.from_numpy(a).cuda() for a in (f, pq, pc)), 10.0).cpu().numpy()
    assert np.abs(got - oracle.relevancy(f, pq, pc, 10.0)).max() <= 1e-5


def test_relevancy_not_finite():
    rng = np.random.default_rng(0)
    f, pq, pc = (rng.normal(size=(m, 40)).astype(np.float32) for m in (70, 3, 2))
    clean = ludvig.relevancy(*(torch.from_numpy(a).cuda() for a in (f, pq, pc)), 10.0).cpu().numpy()
    f[5, 7] = np.nan
    f[6, 7] = np.inf
    got = ludvig.relevancy(*(torch.from_numpy(a).cuda() for a in (f, pq, pc)), 10.0).cpu().numpy()
    rest = [i for i in range(70) if i not in (5, 6)]
    assert np.array_equal(got[rest], clean[rest])
    assert np.all(got[5] == 1.0)   # no phrase compares: the minimum's start
