"""The split iteration (pd_iterate_dual / pd_state_u / pd_iterate_primal) with the data
blocks spread over two shards, both on this GPU in one process: the shards' gridded dual
contributions are summed on the device in place of the all-reduce between GPUs, and
each shard runs the same primal step. The result must match the oracle's single-process
run of Algorithm 1 and the unsplit pd_iterate."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_util import TOL_IT32, TOL_IT64, make_problem, rel  # noqa: E402
from oracle import pd as PD  # noqa: E402
from paper_1610_08895_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import __graft_entry__ as ge
    ge.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_two_shards_match_oracle_and_unsplit_iteration(precision):
    from paper_1610_08895_gb300 import distributed as D
    from paper_1610_08895_gb300.api import Plan, State
    prob, _ = make_problem(128, 30000, 16, 8, (0, 1, 2), 3, uv_kind="radial", blocks="annuli", nannuli=16)
    x0 = synth.start_vector(128, 128, seed=9)
    phi2, psi2 = PD.operator_norms(prob, x0, max_iter=200, tol=1e-8)
    kw = dict(tau=0.49, sigma=1.0 / psi2, varsigma=1.0 / phi2, kappa=1e-3, psi_norm=float(np.sqrt(psi2)), seed=4,
              p_block=[0.5] * 16, p_basis=[0.5] * 3)
    niter = 15
    st_ref, _ = PD.pd_run(prob, niter, **kw)
    cdt = torch.complex64 if precision == "f32" else torch.complex128
    groups = D.shard_blocks(prob.uv, prob.block_of_vis, prob.nblocks, 2)
    shards = []
    for g in groups:
        sh = D.GpuShard(128, 128, prob.uv, prob.block_of_vis, prob.nblocks, g, kw, kernel_width=8,
                        basis_ids=prob.basis_ids, levels=prob.levels, precision=precision)
        sh.set_data(torch.tensor(prob.y[sh.vis], dtype=cdt, device="cuda"), prob.eps)
        shards.append(sh)
    for _ in range(niter):
        for sh in shards:
            sh.dual_step()
        u = shards[0].u_sum_buffer() + shards[1].u_sum_buffer()
        for sh in shards:
            sh.primal_step(u)
    x0_, x1_ = shards[0].x().cpu().numpy(), shards[1].x().cpu().numpy()
    assert np.array_equal(x0_, x1_)                   # the replicated primal update agrees bit for bit
    tol = TOL_IT64 if precision == "f64" else TOL_IT32
    assert rel(x0_, st_ref.x) < tol
    plan = Plan(128, 128, prob.uv, prob.block_of_vis, prob.nblocks, kernel_width=8, basis_ids=prob.basis_ids,
                levels=prob.levels, precision=precision)
    st = State(plan)
    st.pd_state_set_data(torch.tensor(prob.y, dtype=cdt, device="cuda"), prob.eps)
    st.pd_iterate(niter, **kw)
    assert rel(x0_, st.x().cpu().numpy()) < (1e-12 if precision == "f64" else 1e-5)


@pytest.mark.parametrize("precision,J", [("f64", 8), ("f32", 8), ("f32", 12), ("f64", 2)])
def test_state_u_is_the_gridded_dual_sum(precision, J):
    """pd_state_u's grid is G^T v of the oracle, every visibility at its own (u, v), at the same address
    after each call that changes v; pd_iterate_primal takes it or the folded one alike."""
    import ctypes

    from oracle import measurement as meas
    from paper_1610_08895_gb300 import _binding as B
    from paper_1610_08895_gb300 import distributed as D
    from paper_1610_08895_gb300.api import Plan, State
    n, ny, m = 64, 32, 3000
    rng = np.random.default_rng(7)
    uv = rng.uniform(-np.pi, np.pi, size=(m, 2))
    uv[:50] = rng.integers(-32, 32, size=(50, 2)) * (np.pi / 64)          # on grid lines of both axes
    geo = meas.Geometry(ny, n, J)
    plan = Plan(n, ny, uv, (np.arange(m) % 4).astype(np.int32), 4, kernel_width=J, basis_ids=(0, 1), levels=2,
                precision=precision)
    st = State(plan)
    st.pd_state_set_data(torch.tensor(synth.uniform_vis(m, seed=5), dtype=plan.cplx_dtype, device="cuda"), np.ones(4))
    v0 = torch.tensor(synth.uniform_vis(m, seed=6), dtype=plan.cplx_dtype, device="cuda")

    def view(name):
        ptr, k = ctypes.c_void_p(), ctypes.c_int64()
        B.call(name, st._h, ctypes.byref(ptr), ctypes.byref(k))
        typestr = "<c8" if precision == "f32" else "<c16"
        return ptr.value, torch.as_tensor(D._DevArray(ptr.value, k.value, typestr), device="cuda")

    addr, u = view("pd_state_u")
    tol = 1e-12 if precision == "f64" else 1e-5

    def check():
        torch.cuda.synchronize()
        got = u.cpu().numpy().reshape(2 * n // 4, 2 * ny, 4).transpose(1, 0, 2).reshape(2 * ny, 2 * n)
        want = geo.grid(st.v().cpu().numpy().astype(complex), uv).reshape(2 * ny, 2 * n)
        assert rel(got, want) < tol if np.any(want) else not np.any(got)
        assert view("pd_state_u")[0] == addr

    kw = dict(tau=0.49, sigma=1.0, varsigma=1e-4, kappa=1e-3, seed=1, p_block=[0.6] * 4, p_basis=[1.0] * 2)
    check()
    st.pd_state_set_start(v0=v0)
    check()
    buf = st.save()
    for form in (dict(), dict(use_graph=True), dict(per_block=True)):
        st.pd_iterate(3, **kw, **form)
        check()
    st.load(buf)
    check()
    pb, ps = np.full(4, 0.6), np.ones(2)
    prm = B.PdParams(tau=0.49, sigma=1.0, varsigma=1e-4, kappa=1e-3, psi_norm=1.0, seed=1, p_block=pb.ctypes.data,
                     p_basis=ps.ctypes.data)
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    B.call("pd_iterate_dual", plan.handle, st._h, ctypes.byref(prm), stream)
    check()
    after = st.save()
    out = []
    for grid in (None, u.clone(), view("pd_state_u_folded")[1].clone()):
        st.load(after)
        B.call("pd_iterate_primal", plan.handle, st._h, ctypes.byref(prm),
               ctypes.c_void_p(0 if grid is None else grid.data_ptr()), stream)
        out.append(st.x().cpu().numpy())
    assert rel(out[1], out[0]) < tol and rel(out[2], out[0]) < tol
    st.pd_state_set_data(v0, np.ones(4))
    st.pd_synthesis_iterate(2, 0.49, 1.0, 1e-4, 1e-3, seed=1, p_block=[0.6] * 4)
    check()
