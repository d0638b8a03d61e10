"""Groups of views and the forms of the weights pass: launches far above and below the
few-tile limits give the same sums, packed jobs of uneven scenes share groups whose
sorts run ahead, and a call that fails between its groups leaves nothing behind.
Float32 sums of the same terms in another order: 1e-5 relative L2."""
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


@pytest.fixture
def option():
    """Sets options for one test and puts them back."""
    old = {}

    def set_(name, value):
        old.setdefault(name, ludvig.get_option(name))
        ludvig.set_option(name, value)
    yield set_
    for name, value in old.items():
        ludvig.set_option(name, value)


def _same(got, ref):
    assert (ref[1] > 0).any()
    assert rel_l2(got[0].cpu().numpy(), ref[0].cpu().numpy()) <= 1e-5
    assert rel_l2(got[1].cpu().numpy(), ref[1].cpu().numpy()) <= 1e-5


# 9 views of 60 x 34 tiles: 18360 items in one group, then 2040 in each of nine
@pytest.mark.parametrize("d,dtype,count", [(1, torch.float32, False), (4, torch.bfloat16, True), (27, torch.float32, False),
                                           (40, torch.float32, True), (48, torch.bfloat16, False)])
def test_many_and_few_tiles_agree(option, d, dtype, count):
    wl = inputs.small_field_workload(n=20_000, views=9, d=d, width=955, height=539)
    sc = ludvig.Scene.from_inputs(wl.scene)
    F = device_features(wl, range(9), dtype=dtype)
    option(ludvig.OPT_COUNT_NORMALISE, int(count))
    one = ludvig.uplift(sc, wl.cams.params, 955, 539, F)
    option(ludvig.OPT_GROUP_MB, 1)
    _same(ludvig.uplift(sc, wl.cams.params, 955, 539, F), one)


def _faint_slab(n=180_000, seed=11):
    """Faint Gaussians so dense that pixels stay open over hundreds of contributors."""
    rng = np.random.default_rng(seed)
    q = rng.normal(size=(n, 4))
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    return inputs.Scene((rng.uniform(-0.6, 0.6, size=(n, 3)) * [1.0, 1.0, 0.3]).astype(np.float32),
                        np.full((n, 3), 0.03, np.float32), q.astype(np.float32), np.full(n, 0.012, np.float32))


# 9 views of 20 x 15 tiles: 2700 items, whose long lists are handed over, then 300 in each of nine
@pytest.mark.parametrize("d,dtype", [(1, torch.float32), (3, torch.bfloat16), (4, torch.float32), (40, torch.float32),
                                     (48, torch.bfloat16)])
@pytest.mark.parametrize("count", [False, True])
def test_long_lists_handed_over(option, d, dtype, count):
    scene = _faint_slab()
    cams = inputs.cameras_orbit(9, 1.6, 315, 235, 250.0, hemisphere=True)
    sc = ludvig.Scene.from_inputs(scene)
    _, contributors = ludvig.debug_transmittance(sc, cams.params[0], 315, 235)
    open_late = (contributors > 512).float().mean().item()
    assert 0.05 < open_late   # more entries than a warp walks by itself
    F = torch.rand((9, 235, 315, d), device="cuda", generator=torch.Generator("cuda").manual_seed(d)).to(dtype)
    option(ludvig.OPT_COUNT_NORMALISE, int(count))
    one = ludvig.uplift(sc, cams.params, 315, 235, F)
    option(ludvig.OPT_GROUP_MB, 1)
    few = ludvig.uplift(sc, cams.params, 315, 235, F)
    _same(one, few)
    if count:
        assert torch.equal(one[1], few[1])


@pytest.mark.parametrize("d,dtype", [(3, torch.bfloat16), (40, torch.float32), (64, torch.bfloat16)])
def test_packed_jobs_of_uneven_scenes(option, d, dtype):
    option(ludvig.OPT_BATCH_TUNE, 0)
    option(ludvig.OPT_GROUP_MB, 128)
    jobs, ref = [], []
    wls = [inputs.small_field_workload(n=n, views=v, d=d, width=157, height=93)
           for n, v in ((300_000, 7), (20_000, 5), (150_000, 9), (70_000, 12))]
    pool = torch.cat([device_features(wl, range(wl.cams.v), dtype=dtype) for wl in wls])   # (one class: views of one array)
    at = 0
    for wl in wls:
        F = pool[at:at + wl.cams.v]
        at += wl.cams.v
        jobs.append((ludvig.Scene.from_inputs(wl.scene), wl.cams.params, 157, 93, F, None, None))
        ref.append(ludvig.uplift(ludvig.Scene.from_inputs(wl.scene), wl.cams.params, 157, 93, F))
    for _ in range(2):
        for got, r in zip(ludvig.uplift_batch(jobs)[0], ref):
            _same(got, r)


@pytest.mark.parametrize("d,dtype", [(3, torch.bfloat16), (40, torch.float32), (100, torch.float32)])
def test_failure_between_groups_leaves_nothing_running(option, d, dtype):
    """An error that a launch check reports (injected on the host) while other groups'
    work is queued: once it is raised, nothing of the call runs on but what is ordered
    on the caller's stream, so that the caller may use the memory again."""
    wl = inputs.small_field_workload(n=300_000, views=10, d=d, width=157, height=93)
    sc = ludvig.Scene.from_inputs(wl.scene)
    F = device_features(wl, range(10), dtype=dtype)
    option(ludvig.OPT_GROUP_MB, 128)
    ref = ludvig.uplift(sc, wl.cams.params, 157, 93, F)
    out, beta = torch.empty_like(ref[0]), torch.empty_like(ref[1])
    failed = 0
    for k in (20, 33, 45, 52, 60, 71, 84, 97, 110, 125, 140):
        torch.cuda._sleep(20_000_000)   # about 10 ms of SM clock, so that the queue is full when the call fails
        ludvig.set_option(ludvig.OPT_FAULT_LAUNCH, k)
        try:
            ludvig.uplift(sc, wl.cams.params, 157, 93, F, out, beta)
        except ludvig.LudvigError:
            failed += 1
            out.fill_(7.0)   # behind what the call put on this stream
            beta.fill_(7.0)
            torch.cuda.synchronize()
            assert (out == 7.0).all() and (beta == 7.0).all(), k
        finally:
            ludvig.set_option(ludvig.OPT_FAULT_LAUNCH, 0)
        _same(ludvig.uplift(sc, wl.cams.params, 157, 93, F, out, beta), ref)
    assert failed >= 5


@pytest.mark.parametrize("d,dtype", [(3, torch.float32), (40, torch.float32), (48, torch.bfloat16), (100, torch.float32),
                                     (101, torch.bfloat16)])
def test_a_call_that_outgrows_the_workspace_is_redone(d, dtype):
    """A far view sizes the workspace; near ones, in an asynchronous call, need many times
    its pairs and weight rows, with tiles handed over while the rows' capacity is exceeded."""
    scene = _faint_slab()
    far = inputs.cameras_orbit(1, 60.0, 16, 16, 60.0, hemisphere=True)
    near = inputs.cameras_orbit(9, 1.6, 315, 235, 250.0, hemisphere=True)
    F = torch.rand((9, 235, 315, d), device="cuda", generator=torch.Generator("cuda").manual_seed(d)).to(dtype)
    ref = ludvig.uplift(ludvig.Scene.from_inputs(scene), near.params, 315, 235, F)
    sc = ludvig.Scene.from_inputs(scene)
    ludvig.uplift(sc, far.params, 16, 16, F[:1, :16, :16].contiguous())
    small = sc.workspace_bytes()
    _same(ludvig.uplift(sc, near.params, 315, 235, F), ref)
    assert sc.workspace_bytes() > small
    _same(ludvig.uplift(sc, near.params, 315, 235, F), ref)
