"""Several states of one plan: what may run side by side on different streams and threads, and
what each call leaves of the plan's shared scratch to the others."""
import ctypes
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_util import make_problem, rel  # noqa: E402
from paper_1610_08895_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import __graft_entry__ as ge
    ge.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def _plan_and_states(prob, precision, count):
    from paper_1610_08895_gb300.api import Plan, State
    plan = Plan(prob.geom.nx, prob.geom.ny, prob.uv, prob.block_of_vis, prob.nblocks, kernel_width=prob.geom.J,
                basis_ids=prob.basis_ids, levels=prob.levels, precision=precision)
    out = []
    for k in range(count):
        st = State(plan)
        st.pd_state_set_data(torch.tensor((1 + k) * prob.y, dtype=plan.cplx_dtype, device="cuda"), prob.eps)
        out.append(st)
    return plan, out


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_checkpoints_beside_an_iteration_of_another_state(precision):
    """Saving and loading one state while another one of the plan iterates on a second stream: the
    iteration is the one that runs alone, and the buffers are those of the state that was saved."""
    prob, _ = make_problem(128, 40000, 9, 8, (0, 1, 2), 3)
    plan, (a, b) = _plan_and_states(prob, precision, 2)
    kw = dict(tau=0.49, sigma=1.0, varsigma=1e-5, kappa=1e-3, seed=2, p_block=[0.5] * 9, p_basis=[0.5] * 3, use_graph=True)
    v0 = torch.tensor(synth.uniform_vis(len(prob.uv), seed=6), dtype=plan.cplx_dtype, device="cuda")
    b.pd_state_set_start(v0=v0)
    want_b = b.save()
    start = a.save()
    a.pd_iterate(150, **kw)
    want_x, want_v = a.x(), a.v()
    a.load(start)
    one, two = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(one):
        a.pd_iterate(150, **kw)
    with torch.cuda.stream(two):
        for _ in range(10):
            assert np.array_equal(b.save(), want_b)
            b.load(want_b)
    torch.cuda.synchronize()
    assert torch.equal(a.x(), want_x) and torch.equal(a.v(), want_v)
    assert torch.equal(b.v(), v0)


def test_first_checkpoints_from_several_threads():
    """The order of the visibilities is made by a plan's first save: several threads may ask for it."""
    prob, _ = make_problem(128, 60000, 9, 8, (0, 1), 2)
    plan, states = _plan_and_states(prob, "f32", 4)
    bufs = [None] * 4

    def save(k):
        with torch.cuda.stream(torch.cuda.Stream()):
            bufs[k] = states[k].save()

    threads = [threading.Thread(target=save, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for k in range(4):
        assert np.array_equal(bufs[k], states[k].save())
        states[k].load(bufs[k])
        assert np.array_equal(bufs[k], states[k].save())


@pytest.mark.parametrize("kw", [dict(precision="f32"), dict(precision="f64"), dict(precision="f32", g_mode="csr")])
def test_launches_start_from_their_first_item_whatever_an_earlier_one_left(kw):
    """Counters that an earlier launch left anywhere (it overlapped another one, say) do not reach the
    next call: Phi, Phi^H, an iteration and a batch are what they are on untouched counters."""
    from paper_1610_08895_gb300 import _binding as B
    from paper_1610_08895_gb300.api import Plan, State
    n, m = 64, 5000
    uv = synth.uv_gaussian(m, seed=1)
    plan = Plan(n, n, uv, (np.arange(m) % 4).astype(np.int32), 4, basis_ids=(0, 1), levels=2, **kw)
    st = State(plan)
    x = torch.tensor(synth.random_images(2, n, n, seed=3), dtype=plan.real_dtype, device="cuda")
    y = torch.tensor(np.stack([synth.uniform_vis(m, seed=k) for k in (4, 5)]), dtype=plan.cplx_dtype, device="cuda")

    def everything():
        yield plan.pd_apply_phi(x[0])
        yield plan.pd_apply_phi(x)
        yield plan.pd_apply_phi_adj(y[0])
        yield plan.pd_apply_phi_adj(y)
        for form in (dict(), dict(use_graph=True), dict(per_block=True)):
            st.pd_state_set_data(y[0], np.ones(4))
            spoil()
            st.pd_iterate(2, 0.49, 1.0, 1e-4, 1e-3, seed=1, p_block=[0.9] * 4, p_basis=[0.9] * 2, **form)
            yield st.x()
            yield st.v()

    spoil = lambda: None  # noqa: E731
    want = [t.clone() for t in everything()]
    hook = B.load().pd_test_work_counters
    hook.argtypes = [ctypes.c_void_p, ctypes.c_int32]
    spoil = lambda: B.check(hook(plan.handle, 12345))  # noqa: E731
    spoil()
    for got, ref in zip(everything(), want):
        assert rel(got.cpu().numpy(), ref.cpu().numpy()) < 1e-6 and torch.isfinite(torch.view_as_real(got) if got.is_complex() else got).all()
        spoil()
