"""Which kernel variant a call takes: default tiles of a stored G, batches, items with few points."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_util import rel  # noqa: E402
from paper_1610_08895_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import __graft_entry__ as ge
    ge.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def _uv(kind, m):
    if kind == "uniform":
        return np.random.default_rng(3).uniform(-np.pi, np.pi, size=(m, 2))
    return synth.uv_gaussian(m, seed=1) if kind == "gaussian" else synth.uv_radial(m, seed=1)


@pytest.mark.parametrize("n,m,kind,d,dde,tile", [
    (128, 60000, "gaussian", 4, False, 8), (1024, 200000, "uniform", 1, False, 32), (1024, 200000, "radial", 1, True, 32),
    (256, 30000, "radial", 1, True, 16), (1024, 60000, "uniform", 1500, False, 8)])
def test_default_tile_of_a_stored_g_follows_the_points(n, m, kind, d, dde, tile):
    """Large where tiles hold few points, small where the heaviest tile would be all a launch waits for, and
    where so many blocks could share a large one that the plan would be refused; the same operator either way."""
    from paper_1610_08895_gb300.api import Plan
    uv = _uv(kind, m)
    kw = dict(kernel_width=4, g_mode="csr")
    if dde:
        kw["dde_kernels"] = np.random.default_rng(5).normal(size=(m, 3, 3)) + 0j
    blk = (np.arange(m) % d).astype(np.int32)
    plan = Plan(n, n, uv, blk, d, **kw)
    assert plan.info()["tile"] == tile
    other = Plan(n, n, uv, blk, d, tile=16, **kw) if d <= 1024 else plan
    x = torch.tensor(synth.random_images(1, n, n, seed=3)[0], dtype=torch.float32, device="cuda")
    y = plan.pd_apply_phi(x)
    assert rel(other.pd_apply_phi(x).cpu().numpy(), y.cpu().numpy()) < 2e-6
    assert rel(other.pd_apply_phi_adj(y).cpu().numpy(), plan.pd_apply_phi_adj(y).cpu().numpy()) < 2e-6


@pytest.mark.parametrize("n,m,b,kw", [
    (256, 65536, 8, dict()), (64, 5000, 3, dict(kernel_width=6)), (64, 3000, 2, dict(kernel_width=12)),
    (64, 5000, 3, dict(precision="f64")), (64, 5000, 3, dict(g_mode="csr")), (128, 9001, 5, dict(g_mode="csr", precision="f64")),
    (64, 5000, 4, dict(g_mode="csr", kernel_width=6, dde=True))])
def test_a_batch_is_its_images_one_by_one(n, m, b, kw):
    from paper_1610_08895_gb300.api import Plan
    kw = dict(kw)
    if kw.pop("dde", False):
        kw["dde_kernels"] = np.random.default_rng(5).normal(size=(m, 3, 3)) + 0j
    plan = Plan(n, n, _uv("gaussian", m), np.zeros(m, np.int32), 1, **kw)
    x = torch.tensor(synth.random_images(b, n, n, seed=3), dtype=plan.real_dtype, device="cuda")
    v = torch.tensor(np.stack([synth.uniform_vis(m, seed=k) for k in range(b)]), dtype=plan.cplx_dtype, device="cuda")
    y, xa = plan.pd_apply_phi(x), plan.pd_apply_phi_adj(v)
    for k in range(b):
        assert torch.equal(y[k], plan.pd_apply_phi(x[k].contiguous()))
        one = plan.pd_apply_phi_adj(v[k].contiguous())
        if "g_mode" in kw or kw.get("precision") == "f64":
            assert torch.equal(xa[k], one)
        else:       # a batch's tiles may be shared out to other warps; J > 8 adds through shared-memory atomics
            assert rel(xa[k].cpu().numpy(), one.cpu().numpy()) < 2e-6
    if kw.get("kernel_width", 8) <= 8:
        assert torch.equal(xa, plan.pd_apply_phi_adj(v))


@pytest.mark.parametrize("J", [8, 12])
def test_residual_norms_where_items_hold_few_points(J):
    """2,000 items of some 50 points, worked on by smaller blocks, with many blocks of data to an item."""
    from oracle import measurement as meas
    from paper_1610_08895_gb300.api import Plan, State
    n, m, d = 512, 100001, 37
    uv = _uv("uniform", m)
    blk = (np.arange(m) % d).astype(np.int32)
    plan = Plan(n, n, uv, blk, d, kernel_width=J)
    x = synth.random_images(1, n, n, seed=3)[0]
    y = synth.uniform_vis(m, seed=4)
    want = meas.Geometry(n, n, J).phi(x, uv)
    xt = torch.tensor(x, dtype=torch.float32, device="cuda")
    assert rel(plan.pd_apply_phi(xt).cpu().numpy(), want) < 1e-5
    st = State(plan)
    st.pd_state_set_data(torch.tensor(y, dtype=torch.complex64, device="cuda"), np.ones(d))
    st.pd_state_set_start(x0=xt)
    norms = np.sqrt(np.bincount(blk, weights=np.abs(want - y) ** 2, minlength=d))
    assert np.max(np.abs(st.report()["res_norm"] / norms - 1)) < 1e-5


@pytest.mark.parametrize("n,tile,d", [(2048, 8, 256), (64, 8, 7), (64, 64, 1)])
def test_order_of_the_points(n, tile, d):
    """Plans whose (tile, block) pairs are too many for one counting pass (262,144 tiles, 256 blocks), and segments
    with many and with few points to a cell: Phi, Phi^H and a checkpoint read back."""
    from paper_1610_08895_gb300.api import Plan, State
    m = 20011
    uv = _uv("gaussian", m)
    uv[:4000] = uv[:40].repeat(100, axis=0)                     # ties, which stay in the order they came in
    blk = (np.arange(m) * 31 % d).astype(np.int32)
    plan, other = Plan(n, n, uv, blk, d, tile=tile), Plan(n, n, uv, blk, d, tile=16)
    x = torch.tensor(synth.random_images(1, n, n, seed=3)[0], dtype=torch.float32, device="cuda")
    y = plan.pd_apply_phi(x)
    assert rel(other.pd_apply_phi(x).cpu().numpy(), y.cpu().numpy()) < 2e-6
    assert rel(other.pd_apply_phi_adj(y).cpu().numpy(), plan.pd_apply_phi_adj(y).cpu().numpy()) < 2e-6
    st = State(plan)
    st.pd_state_set_data(y, np.ones(d))
    st.pd_state_set_start(v0=y)
    buf = st.save()
    st.pd_state_set_data(y, np.ones(d))
    st.load(buf)
    assert torch.equal(st.v(), y)


@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_autotuner_offers_the_tile_that_a_plan_would_choose(precision):
    from paper_1610_08895_gb300.api import Plan, autotune_tile
    n, m = 64, 3000
    uv, blk = _uv("gaussian", m), np.zeros(m, np.int32)
    best, times = autotune_tile(n, n, uv, blk, 1, precision=precision, iters=1)
    assert Plan(n, n, uv, blk, 1, precision=precision).info()["tile"] in times
    assert times[best] == min(t for t in times.values() if t > 0)
