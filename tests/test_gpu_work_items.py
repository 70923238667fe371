"""Points at the edges of the gridding's and degridding's work items: one point, chunks of 32
with a remainder, a tile so heavy that it is split into parts, points on grid lines and at
the band edges (which are not held as conjugates), every kernel width and tile size; the
fixed order of the sums; the order in which a checkpoint keeps the visibilities."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_util import TOL_OP32, TOL_OP64, rel  # noqa: E402
from oracle import measurement as meas  # noqa: E402
from paper_1610_08895_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import __graft_entry__ as ge
    ge.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def _points(kind, m, n, seed=0):
    rng = np.random.default_rng(seed)
    if kind == "cluster":           # all in one tile
        return np.array([0.7, -1.1]) + rng.uniform(0.0, 6.0 * np.pi / n, size=(m, 2))
    if kind == "lines":             # integer grid coordinates in x, in y, in both, and the band edges
        k = rng.integers(-n, n, size=(m, 2)) * (np.pi / n)
        f = rng.uniform(-np.pi, np.pi, size=(m, 2))
        uv = np.where(rng.integers(0, 2, size=(m, 2)) == 0, k, f)
        uv[:4] = [[-np.pi, -np.pi], [0.0, 0.0], [-np.pi, 0.3], [0.3, -np.pi]]
        return uv
    return synth.uv_gaussian(m, seed=seed + 1)


CASES = [
    # kind, m, n, blocks, J, tile
    ("gauss", 1, 16, 1, 8, 0), ("gauss", 31, 16, 2, 6, 8), ("gauss", 33, 32, 3, 4, 16), ("gauss", 65, 32, 1, 2, 2),
    ("gauss", 4097, 64, 5, 8, 8), ("gauss", 3000, 64, 7, 8, 64), ("lines", 2000, 32, 4, 8, 16),
    ("lines", 1500, 32, 2, 6, 8), ("lines", 1200, 32, 3, 4, 32), ("lines", 700, 32, 1, 2, 16),
    ("cluster", 9001, 64, 3, 8, 16), ("cluster", 8500, 128, 40, 6, 32), ("cluster", 3001, 64, 2, 12, 16),
]


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("case", CASES)
def test_operators_at_the_edges_of_work_items(case, precision):
    from paper_1610_08895_gb300.api import Plan
    kind, m, n, nb, J, tile = case
    if kind == "lines" and precision == "f32" and J <= 4:
        pytest.skip("the kernel's jump at |t| = J/2 is above FP32 rounding: a fraction that rounds to a grid "
                    "line takes another set of taps than the FP64 oracle")
    uv = _points(kind, m, n)
    geo = meas.Geometry(n, n, J)
    plan = Plan(n, n, uv, (np.arange(m) % nb).astype(np.int32), nb, kernel_width=J, precision=precision, tile=tile)
    x = synth.random_images(1, n, n, seed=3)[0]
    v = synth.uniform_vis(m, seed=4)
    tol = TOL_OP32 if precision == "f32" else TOL_OP64
    y = plan.pd_apply_phi(torch.tensor(x, dtype=plan.real_dtype, device="cuda")).cpu().numpy()
    assert rel(y, geo.phi(x, uv)) < tol
    vt = torch.tensor(v, dtype=plan.cplx_dtype, device="cuda")
    xa = plan.pd_apply_phi_adj(vt)
    assert rel(xa.cpu().numpy(), geo.phi_adj(v, uv)) < tol
    if J <= 8:                      # wider kernels add through shared-memory atomics
        assert torch.equal(xa, plan.pd_apply_phi_adj(vt))


@pytest.mark.parametrize("tile", [0, 16])
def test_checkpoint_order_of_the_visibilities(tile):
    """The buffer holds v by (tile, block, 8 x 8 super-cell, row, column, user index) of the base cells."""
    from paper_1610_08895_gb300.api import Plan, State
    n, m, nb, J = 64, 3000, 5, 8
    uv = _points("lines", m, n, seed=2)
    blk = (np.arange(m) % nb).astype(np.int32)
    plan = Plan(n, n, uv, blk, nb, kernel_width=J, precision="f64", tile=tile)
    st = State(plan)
    st.pd_state_set_data(torch.tensor(synth.uniform_vis(m, seed=5), device="cuda"), np.ones(nb))
    v0 = synth.uniform_vis(m, seed=6)
    st.pd_state_set_start(v0=torch.tensor(v0, device="cuda"))
    buf = st.save()
    N, T = n * n, tile or 32
    start = 8 * (2 * N + plan.nbases * N + N)
    got = buf[start:start + 16 * m].view(np.complex128)
    base = np.floor(uv * (2 * n) / (2 * np.pi)).astype(np.int64) % (2 * n)
    bx, by = base[:, 0], base[:, 1]
    sc = (by % T) // 8 * (T // 8) + (bx % T) // 8
    order = np.lexsort((np.arange(m), bx, by, sc, blk, (by // T) * (2 * n // T) + bx // T))
    assert np.array_equal(got, v0[order])
    other = State(plan)
    other.load(buf)
    assert np.array_equal(other.v().cpu().numpy(), v0)


@pytest.mark.parametrize("n,levels", [(16, 2), (32, 1), (64, 3), (128, 2), (256, 4)])
def test_dictionary_on_buffers_that_start_anywhere(n, levels):
    """Psi^H and Psi on 4-byte aligned buffers equal the aligned ones: the 16-byte kernels and
    the general ones they give way to (and each of their tile sizes) compute the same filters."""
    from paper_1610_08895_gb300.api import Plan
    ids = (0, 1, 2, 5, 8)
    plan = Plan(n, n, np.zeros((1, 2)), np.zeros(1, np.int32), 1, basis_ids=ids, levels=levels)
    x = torch.tensor(synth.random_images(1, n, n, seed=1)[0], dtype=torch.float32, device="cuda")
    big = torch.zeros(n * n + 1, dtype=torch.float32, device="cuda")
    odd = big[1:].view(n, n)
    odd.copy_(x)
    a = plan.pd_apply_psi_adj(x)
    coeffs = torch.zeros(a.numel() + 1, dtype=torch.float32, device="cuda")[1:].view_as(a)
    b = plan.pd_apply_psi_adj(odd, coeffs)
    assert rel(b.cpu().numpy(), a.cpu().numpy()) < 2e-6        # 2 x 16 taps a level, summed in another order
    back = plan.pd_apply_psi(b, torch.zeros(n * n + 1, dtype=torch.float32, device="cuda")[1:].view(n, n))
    assert rel(back.cpu().numpy(), x.cpu().numpy()) < TOL_OP32
    assert rel(plan.pd_apply_psi(a).cpu().numpy(), x.cpu().numpy()) < TOL_OP32


def _hold(plan, polls, hold):
    import ctypes
    from paper_1610_08895_gb300 import _binding as B
    hook = B.load().pd_test_ordered_adds
    hook.argtypes = [ctypes.c_void_p, ctypes.c_int32, ctypes.c_int32]
    B.check(hook(plan.handle, polls, hold))


def _timeout(call):
    from paper_1610_08895_gb300 import _binding as B
    with pytest.raises(B.PDError) as e:
        call()
    return e.value.status == B.PD_ETIMEOUT


def test_a_wait_of_the_ordered_adds_that_gives_up():
    """A short limit and one part too many pending: the launch ends, the sums are complete, every state
    keeps its own flag until its data are set anew, plain applications theirs, and the next call
    is as if nothing had been."""
    from paper_1610_08895_gb300.api import Plan, State
    n, m, nb, J = 64, 6000, 4, 8
    uv = _points("gauss", m, n)
    geo = meas.Geometry(n, n, J)
    plan = Plan(n, n, uv, (np.arange(m) % nb).astype(np.int32), nb, kernel_width=J, basis_ids=(0, 1), levels=2)
    v = synth.uniform_vis(m, seed=4)
    vt = torch.tensor(v, dtype=plan.cplx_dtype, device="cuda")
    kw = dict(tau=0.49, sigma=1.0, varsigma=1e-4, kappa=1e-3, seed=1, p_block=[1.0] * nb, p_basis=[1.0] * 2)
    a, b = State(plan), State(plan)
    for st in (a, b):
        st.pd_state_set_data(vt, np.ones(nb))
    want = plan.pd_apply_phi_adj(vt)
    a.pd_iterate(3, **kw)
    want_x, start = a.x(), b.save()
    a.report()
    plan.pd_plan_status()
    a.pd_state_set_data(vt, np.ones(nb))
    _hold(plan, 8, 1)
    for form in (dict(), dict(use_graph=True), dict(per_block=True)):
        a.pd_state_set_data(vt, np.ones(nb))
        a.report()
        a.pd_iterate(3, **kw, **form)
        assert rel(a.x().cpu().numpy(), want_x.cpu().numpy()) < 1e-5      # complete; another order of the sums
        assert _timeout(a.report) and _timeout(a.report)
    plan.pd_plan_status()                                                   # not a plain application's
    xa = plan.pd_apply_phi_adj(vt)
    assert rel(xa.cpu().numpy(), geo.phi_adj(v, uv)) < TOL_OP32
    assert _timeout(plan.pd_plan_status)
    x0 = torch.tensor(synth.random_images(1, n, n, seed=3)[0], dtype=plan.real_dtype, device="cuda")
    assert _timeout(lambda: plan.pd_operator_norms(x0, 3, 0.0))
    b.report()                                                              # nor another state's
    assert _timeout(lambda: b.pd_state_set_start(v0=vt)) and _timeout(b.report)
    _hold(plan, 1 << 22, 0)
    assert torch.equal(plan.pd_apply_phi_adj(vt), want)
    assert _timeout(a.report)
    b.load(start)
    b.report()
    a.pd_state_set_data(vt, np.ones(nb))
    a.pd_iterate(3, **kw)
    assert a.report()["t"] == 3 and torch.equal(a.x(), want_x)


@pytest.mark.parametrize("precision,form", [("f32", dict()), ("f32", dict(use_graph=True)), ("f32", dict(per_block=True)),
                                            ("f64", dict()), ("f64", dict(per_block=True))])
def test_iterations_with_a_tile_that_is_split_into_parts(precision, form):
    """9,001 points in one tile of 16 cells (three gridding and nine degridding parts) and 400 around it,
    in blocks of which few are active: parts left without a point, shares that differ from the slots'
    ranges, and neighbours that add to the same cells. Against the oracle, and twice the same bits."""
    from gpu_util import TOL_IT32, TOL_IT64
    from oracle import pd as PD
    from paper_1610_08895_gb300.api import Plan, State
    n, nb, J = 64, 11, 8
    rng = np.random.default_rng(5)
    g = np.concatenate([np.array([20.0, 36.0]) + rng.uniform(0.0, 12.0, size=(9001, 2)),      # one tile's cells
                        np.array([10.0, 26.0]) + rng.uniform(0.0, 32.0, size=(400, 2))])
    uv = g * (np.pi / n)
    blk = np.sort(rng.integers(0, nb, size=len(uv))).astype(np.int32)
    blk[9001:] = rng.integers(0, nb, size=400)
    prob = PD.Problem(meas.Geometry(n, n, J), uv, blk, nb, [0, 1, 2], 2)
    phix = prob.phi(synth.test_image(n, seed=2))
    prob.y = phix + 0.05 * np.abs(phix).mean() * synth.complex_noise(len(uv), seed=3)
    prob.eps = np.array([0.05 * np.abs(phix).mean() * np.sqrt(max(len(ix), 1)) for ix in prob.block_index])
    kw = dict(tau=0.49, sigma=1.0, varsigma=1.0 / (9001 * n * n / 4.0), kappa=1e-3, psi_norm=1.0, seed=6,
              p_block=[0.3] * nb, p_basis=[0.7] * 3)
    ref, draws = PD.pd_run(prob, 12, **kw)
    assert min(sum(d[0]) for d in draws) <= 2                                   # few active blocks at times
    plan = Plan(n, n, uv, blk, nb, kernel_width=J, basis_ids=[0, 1, 2], levels=2, precision=precision, tile=16)
    out = []
    for _ in range(2):
        st = State(plan)
        st.pd_state_set_data(torch.tensor(prob.y, dtype=plan.cplx_dtype, device="cuda"), prob.eps)
        st.pd_iterate(12, **kw, **form)
        out.append((st.x(), st.s(), st.v()))
        rep = st.report()
    assert all(torch.equal(a, b) for a, b in zip(*out))
    tol = TOL_IT64 if precision == "f64" else TOL_IT32
    assert rel(out[0][0].cpu().numpy(), ref.x) < tol and rel(out[0][2].cpu().numpy(), ref.v) < tol
    # s holds small differences of much larger analysis coefficients, whose rounding is relative to them
    scale = np.linalg.norm(prob.psi_adj(ref.x_tilde))
    assert np.linalg.norm(out[0][1].cpu().numpy() - ref.s) < (TOL_IT64 if precision == "f64" else 1e-5) * scale
    assert list(rep["block_active"]) == list(draws[-1][0])
