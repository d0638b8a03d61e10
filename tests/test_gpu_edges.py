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


def _uplift_error(wl, dtype, count=False):
    sc = ludvig.Scene.from_inputs(wl.scene)
    F = device_features(wl, range(wl.cams.v), dtype=dtype)
    old = ludvig.get_option(ludvig.OPT_COUNT_NORMALISE)
    ludvig.set_option(ludvig.OPT_COUNT_NORMALISE, int(count))
    try:
        out, beta = ludvig.uplift(sc, wl.cams.params, wl.cams.width, wl.cams.height, F)
    finally:
        ludvig.set_option(ludvig.OPT_COUNT_NORMALISE, old)
    ref, bref = oracle.uplift(wl.scene, wl.cams, lambda v: F[v].float(), count_normalise=count)
    pos = bref > 0
    assert np.array_equal(beta.cpu().numpy() > 0, pos)
    if count:
        assert np.array_equal(beta.cpu().numpy(), bref)
    return rel_l2(out.cpu().numpy(), ref, pos)


# 5 views of 30 x 17 tiles: 2550 items, above the few-tile kernels' limits
@pytest.mark.parametrize("d,dtype,gate,count", [(1, torch.float32, 1e-5, False), (3, torch.bfloat16, 1e-2, False),
                                                (4, torch.float32, 1e-5, True), (40, torch.float32, 1e-5, False),
                                                (40, torch.bfloat16, 1e-2, False), (48, torch.float32, 1e-5, True)])
def test_many_tiles(d, dtype, gate, count):
    wl = inputs.small_field_workload(n=6000, views=5, d=d, width=475, height=269)
    assert _uplift_error(wl, dtype, count) <= gate


# groups of 3, 3, 3 and 1 views whose depth sorts (74 tiles of keys a view) take the
# several-block scan and run beside the group before; two calls, the second on a sized
# workspace.  Sums of float32 in another order: the bar is the float32 uplift's.
@pytest.mark.parametrize("d,dtype", [(3, torch.bfloat16), (40, torch.float32), (100, torch.float32)])
def test_groups_sorted_ahead(d, dtype):
    wl = inputs.small_field_workload(n=300_000, views=10, d=d, width=157, height=93)
    sc = ludvig.Scene.from_inputs(wl.scene)
    F = device_features(wl, range(10), dtype=dtype)
    one, b1 = ludvig.uplift(sc, wl.cams.params, wl.cams.width, wl.cams.height, F)
    saved = ludvig.get_option(ludvig.OPT_GROUP_MB)
    ludvig.set_option(ludvig.OPT_GROUP_MB, 128)
    try:
        for _ in range(2):
            many, bm = ludvig.uplift(sc, wl.cams.params, wl.cams.width, wl.cams.height, F)
            assert rel_l2(many.cpu().numpy(), one.cpu().numpy()) <= 1e-5
            assert rel_l2(bm.cpu().numpy(), b1.cpu().numpy()) <= 1e-5
    finally:
        ludvig.set_option(ludvig.OPT_GROUP_MB, saved)


# weights of the CUDA-core path are float32, so bfloat16 features meet the float32 bar
@pytest.mark.parametrize("d,dtype,count", [(33, torch.float32, False), (100, torch.float32, False),
                                           (101, torch.bfloat16, False), (132, torch.float32, True),
                                           (516, torch.bfloat16, False), (520, torch.float32, False)])
def test_cuda_core_widths(d, dtype, count):
    wl = inputs.small_field_workload(n=20_000, views=2, d=d, width=83, height=61)
    assert _uplift_error(wl, dtype, count) <= 1e-5


def test_cuda_core_features_not_finite():
    """A Gaussian without weight at a pixel does not see what the pixel holds."""
    wl = inputs.small_field_workload(n=3000, views=1, d=33, width=83, height=61)
    sc = ludvig.Scene.from_inputs(wl.scene)
    F = device_features(wl, [0])
    out, _ = ludvig.uplift(sc, wl.cams.params, 83, 61, F)
    hit = torch.zeros((1, 61, 83, 1), device="cuda")
    hit[0, 30, 40] = 1.0
    touched, _ = ludvig.uplift(sc, wl.cams.params, 83, 61, hit)
    F[0, 30, 40] = float("nan")
    F[0, 30, 40, 1] = float("inf")
    bad, _ = ludvig.uplift(sc, wl.cams.params, 83, 61, F)
    t = touched[:, 0] > 0
    assert t.any() and torch.isnan(bad[t][:, 0]).all()
    assert torch.isfinite(bad[~t]).all()
    assert rel_l2(bad[~t].cpu().numpy(), out[~t].cpu().numpy()) <= 1e-5


def test_fp8_cuda_core_width():
    """Codes of a width the tensor cores do not take are decoded first."""
    wl = inputs.small_field_workload(n=5000, views=2, d=36, width=61, height=45)
    sc = ludvig.Scene.from_inputs(wl.scene)
    q, s = ludvig.fp8_quantize(device_features(wl, range(2)))
    x = (q.view(torch.float8_e4m3fn).float() * s.view(-1, 1, 1, 1)).bfloat16()
    out, _ = ludvig.uplift_fp8(sc, wl.cams.params, 61, 45, q, s)
    ref, _ = ludvig.uplift(sc, wl.cams.params, 61, 45, x.contiguous())
    assert rel_l2(out.cpu().numpy(), ref.cpu().numpy()) <= 1e-6


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


def _graph_ref(n, k, df, seed):
    s = inputs.scene_clusters(n, seed=seed, n_clusters=5, sigma=0.05, extent=1.0)
    f = np.random.default_rng(seed).normal(size=(n, df)).astype(np.float32)
    f[::97] = 0.0
    nbr, _ = oracle.knn(s.means, k)
    return s, f, nbr, oracle.union_edges(nbr)


@pytest.mark.parametrize("n,k,df", [(40, 3, 1), (20_000, 8, 127), (3000, 16, 128), (3000, 5, 132), (2000, 16, 390),
                                    (2000, 33, 512), (1500, 4, 515)])
def test_graph_widths(n, k, df):
    s, f, nbr, (rows, cols) = _graph_ref(n, k, df, n + df)
    sc = ludvig.Scene.from_inputs(s)
    assert np.array_equal(ludvig.knn(sc, k).cpu().numpy(), nbr)
    g = ludvig.Graph(sc, k, torch.from_numpy(f).cuda(), spatial_h=0.01, row_normalize=True)
    _, col, val = (t.cpu().numpy() for t in g.export())
    A = oracle.csr(n, rows, cols, oracle.edge_weights_spatial_cos(s.means, f, rows, cols, h=0.01))
    assert np.array_equal(col, cols)
    assert rel_l2(val, np.asarray(A[rows, cols]).ravel()) <= 1e-5


@pytest.mark.parametrize("dx,scale", [(2, 1.0), (4, 1e-30), (5, 1e25), (17, 1.0), (32, 1e-12)])
def test_diffusion_columns(dx, scale):
    """Column remainders; the norms hold over the float32 range."""
    s, f, _, (rows, cols) = _graph_ref(5000, 8, 16, dx)
    sc = ludvig.Scene.from_inputs(s)
    g = ludvig.Graph(sc, 8, torch.from_numpy(f).cuda(), spatial_h=0.01, row_normalize=True)
    A = oracle.csr(5000, rows, cols, oracle.edge_weights_spatial_cos(s.means, f, rows, cols, h=0.01))
    x = (np.random.default_rng(dx).random((5000, dx)) * scale).astype(np.float32)
    x[:, 0] = 0.0
    for steps, gate in ((1, 1e-5), (6, 1e-4)):
        got = g.diffuse(torch.from_numpy(x).cuda(), steps).cpu().numpy()
        ref = oracle.diffuse(A, x, steps)
        assert np.all(got[:, 0] == 0.0)
        for c in range(1, dx):
            assert rel_l2(got[:, c], ref[:, c]) <= gate
