"""How far G^T v (read through pd_state_u) is from 64-bit arithmetic, beyond the operators' tolerances."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import measurement as meas  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import __graft_entry__ as ge
    ge.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def _gridded(nx, ny, uv, v, J, precision):
    """G^T v as [2 ny, 2 nx], gridded by the library."""
    from paper_1610_08895_gb300 import _binding as B
    from paper_1610_08895_gb300 import distributed as D
    from paper_1610_08895_gb300.api import Plan, State
    plan = Plan(nx, ny, uv, np.zeros(len(uv), np.int32), 1, kernel_width=J, precision=precision)
    st = State(plan)
    vt = torch.tensor(v, dtype=plan.cplx_dtype, device="cuda")
    st.pd_state_set_data(vt, np.ones(1))
    st.pd_state_set_start(v0=vt)
    ptr, k = ctypes.c_void_p(), ctypes.c_int64()
    B.call("pd_state_u", st._h, ctypes.byref(ptr), ctypes.byref(k))
    torch.cuda.synchronize()
    u = torch.as_tensor(D._DevArray(ptr.value, k.value, "<c8" if precision == "f32" else "<c16"), device="cuda")
    return u.cpu().numpy().reshape(2 * nx // 4, 2 * ny, 4).transpose(1, 0, 2).reshape(2 * ny, 2 * nx)


@pytest.mark.parametrize("J", [4, 6, 8])
def test_fp32_gridding_has_no_bias(J):
    """Roundings to nearest (2^-24 at most each) have no common sign: over some 10^4 cells and four draws the
    projection of G^T v on the exact one is off by less than 1e-9 of it, and a sixth of 2^-24 leaves room
    for the products that the three-way split drops. Sums that the tensor cores truncate are 2e-8 short."""
    scales = []
    for seed in range(4):
        rng = np.random.default_rng(seed)
        uv = rng.uniform(-2.5, 2.5, size=(20000, 2))
        uv[:, 0] = np.abs(uv[:, 0]) + 0.3
        v = rng.normal(size=20000).astype(np.float32) + 0j
        ref = meas.Geometry(64, 64, J).grid(v, uv)
        got = _gridded(64, 64, uv, v, J, "f32").astype(np.complex128)
        scales.append((np.vdot(ref, got) / np.vdot(ref, ref)).real - 1.0)
        assert np.linalg.norm(got - ref) / np.linalg.norm(ref) < 1.2e-7      # two units of rounding
    assert abs(np.mean(scales)) < 1e-8, scales


def _kb(t, J, beta):
    """I0(beta sqrt(1 - (2 t / J)^2)) by its power series in extended precision."""
    s = 1 - (2 * t / J) ** 2
    q, term, out = np.longdouble(beta) ** 2 / 4, np.ones_like(s), np.ones_like(s)
    for k in range(1, 400):
        term = term * q * s / (np.longdouble(k) * k)
        out = out + term
        if np.all(term < out * 1e-22):
            break
    return np.where(s > 0, out, 0)


@pytest.mark.parametrize("J", [2, 4, 6, 8, 10, 16])
def test_fp64_taps_are_exact_to_themselves(J):
    """G^T of single points in FP64 plans: every cell of the footprint to 1e-13 of its own value, the outermost
    ones (some 1e-14 of the largest at J = 8) included. Two taps of at most 20 roundings of 1.1e-16 each; the
    oracle's own argument rounding is up to beta^2 / 2 * 1.1e-16 = 8e-14 there, so the weights are taken
    in extended precision."""
    beta = np.longdouble(meas.kb_beta_default(J, 2.0))
    rng = np.random.default_rng(J)
    n = 32
    for fx, fy in [(0.5, 0.25), (1e-6, 1 - 1e-6), (0.999, 0.001)] + [tuple(rng.random(2)) for _ in range(4)]:
        g = np.array([5 + fx, 9 + fy])
        uv = (g * (np.pi / n))[None]
        got = _gridded(n, n, uv, np.array([1.0 + 0j]), J, "f64")
        g = (uv[0] * 2 * n / (2.0 * np.pi)).astype(np.longdouble)        # as the plan rounds it
        base = np.floor(g).astype(int)
        cells = [(base[k] - J // 2 + 1 + np.arange(J)) for k in range(2)]
        w = [_kb(g[k] - cells[k], J, beta) for k in range(2)]
        want = np.outer(w[1], w[0])
        have = got[np.ix_(cells[1] % (2 * n), cells[0] % (2 * n))]
        assert np.all(have.imag == 0)
        assert np.max(np.abs(have.real / want - 1)) < 1e-13
