"""The work that users of this package have it do, as cases that can be timed and checked.

Every case goes through the public Python entry points (``Plan``, ``State``,
``autograd.phi``, ``psi_adj_noalloc``) the way an imaging program calls them. Four kinds:

* ``phi``: y = Phi x and, for a gradient g, Re(Phi^H g), through ``torch.autograd`` (one
  forward and one backward application, alone or for a batch of images);
* ``psi``: analysis of an image in all bases and synthesis of a set of coefficients;
* ``pd``: the measurements are loaded and Algorithm 1 runs for a number of iterations;
* ``synth``: the same for the synthesis formulation.

Inputs are synthetic: an image of Gaussian blobs and point sources, whose visibilities
have a closed form, with 30 dB of noise; uv points of a Gaussian or a radial coverage;
blocks of equal counts or annuli cut into sectors.
"""
import math

import numpy as np
import torch

from paper_1610_08895_gb300 import autograd
from paper_1610_08895_gb300.api import Plan, State, psi_adj_noalloc

DEV = "cuda"
STEP = dict(tau=0.49, sigma=1.0, kappa=0.05)

PHI = dict(kind="phi", nx=64, ny=64, m=4096, uv="gaussian", width=8, precision="f32", batch=0)
PSI = dict(kind="psi", nx=64, ny=64, bases=9, levels=4, precision="f32", noalloc=False)
PD = dict(kind="pd", nx=64, ny=64, m=4096, uv="gaussian", nblocks=4, width=8, dde=0, csr=False, bases=9, levels=4,
          precision="f32", iters=10, graph=False, adaptive=False, weights=False, p=0.5)
SYNTH = dict(kind="synth", nx=64, ny=64, m=4096, uv="gaussian", nblocks=4, width=8, dde=0, csr=False, bases=9,
             levels=4, precision="f32", iters=4, p=0.5)


def listed():
    return [
        # a gradient step on a small image (the size of the shortest reconstructions): launch latency
        dict(PHI, name="phi_64", width=4),
        # a rectangular image, a number of points that nothing divides, a narrower kernel
        dict(PHI, name="phi_512x256_ragged", nx=512, ny=256, m=99991, uv="radial", width=6),
        # the operators in double precision, for validation runs
        dict(PHI, name="phi_256_f64", nx=256, ny=256, m=65536, precision="f64"),
        # training through Phi: a batch of eight images, 4.2 million visibilities each
        dict(PHI, name="phi_1024_batch8", nx=1024, ny=1024, m=4194304, batch=8),
        # the dictionary alone on the largest image of the benchmark
        dict(PSI, name="psi_2048", nx=2048, ny=2048),
        # a small reconstruction (16 equal blocks, half of them drawn), graph replay: latency of an iteration
        dict(PD, name="pd_256", nx=256, ny=256, m=65536, nblocks=16, iters=25, graph=True),
        # a million visibilities in 64 uneven annuli with adaptive probabilities
        dict(PD, name="pd_512_adaptive", nx=512, ny=512, m=1048576, uv="radial", nblocks=64, graph=True, adaptive=True),
        # the benchmark's problem: 2048^2 image, 16.8 million visibilities, 256 blocks
        dict(PD, name="pd_2048", nx=2048, ny=2048, m=16777216, uv="radial", nblocks=256, iters=6, graph=True),
        # an outer step of the reweighted prior: weights from the current image, then iterations, default options
        dict(PD, name="pd_512_reweighted", nx=512, ny=512, m=300007, nblocks=16, iters=8, weights=True),
        # G stored as a sparse matrix
        dict(PD, name="pd_1024_csr", nx=1024, ny=1024, m=4194304, nblocks=64, iters=4, csr=True),
        # direction-dependent effects: a 3 x 3 kernel per visibility convolved into the rows of G
        dict(PD, name="pd_512_dde", nx=512, ny=512, m=1048576, uv="radial", nblocks=64, width=6, dde=3, csr=True,
             iters=5),
        # the synthesis formulation
        dict(SYNTH, name="synth_1024", nx=1024, ny=1024, m=2097152, nblocks=64),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["phi", "phi", "psi", "pd", "pd", "pd", "pd", "synth"])
    f64 = rng.random() < 0.15
    top = 9 if f64 else 10
    nx, ny = 2 ** rng.randint(6, top), 0
    ny = nx if rng.random() < 0.6 else 2 ** rng.randint(6, top)
    c = dict({"phi": PHI, "psi": PSI, "pd": PD, "synth": SYNTH}[kind], nx=nx, ny=ny, precision="f64" if f64 else "f32")
    if kind == "psi":
        c.update(bases=rng.randint(2, 9), levels=rng.randint(2, 5), noalloc=max(nx, ny) <= 256 and rng.random() < 0.5)
        return c
    c.update(m=logint(1000, min(4000000, 16 * nx * ny) // (10 if f64 else 1)) | 1, uv=rng.choice(["gaussian", "radial"]),
             width=rng.choice([4, 6, 8, 8, 8]))
    if kind == "phi":
        c.update(batch=rng.choice([0, 0, 0, 2, 3, 5, 8]))
        if c["batch"]:
            c["m"] = c["m"] // c["batch"] | 1
        return c
    c.update(nblocks=rng.choice([4, 9, 16, 49, 64, 256]), bases=rng.choice([2, 5, 9, 9, 9]), levels=rng.randint(2, 5),
             iters=logint(1, 20), p=round(rng.uniform(0.25, 1.0), 3))
    if rng.random() < 0.3:
        c.update(csr=True)
        if c["width"] < 8 and rng.random() < 0.5:
            c.update(dde=3)
    if kind == "pd":
        c.update(graph=rng.random() < 0.6, adaptive=rng.random() < 0.25, weights=rng.random() < 0.25)
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed, k):
    return torch.Generator(device=DEV).manual_seed(1000003 * int(seed) + k)


def _uv(case, seed):
    """[m, 2] points in [-pi, pi)^2: radial (inner density 8 x the outer) or a clipped Gaussian."""
    m, g = case["m"], _gen(seed, 1)
    if case["uv"] == "radial":
        n = 5 * m + 1000
        r = math.pi * torch.sqrt(torch.rand(n, generator=g, device=DEV, dtype=torch.float64))
        th = 2.0 * math.pi * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
        keep = torch.rand(n, generator=g, device=DEV, dtype=torch.float64) < 8.0 ** (-r / math.pi)
        p = torch.stack([r * torch.cos(th), r * torch.sin(th)], dim=1)[keep]
    else:
        p = 0.25 * math.pi * torch.randn(m + m // 50 + 1000, 2, generator=g, device=DEV, dtype=torch.float64)
    p = p[((p >= -math.pi) & (p < math.pi)).all(dim=1)][:m]
    if p.shape[0] != m:
        raise RuntimeError("too few points drawn")
    return p.contiguous()


def _blocks(case, uv):
    """Block of each point: radial coverages in annuli (cut into 8 sectors from 128 blocks on),
    Gaussian ones in equal counts (strips in u, each cut in v)."""
    d, m = case["nblocks"], uv.shape[0]
    if case["uv"] == "radial":
        sectors = 8 if d >= 128 else 1
        ring = torch.clamp((torch.hypot(uv[:, 0], uv[:, 1]) / math.pi * (d // sectors)).long(), max=d // sectors - 1)
        sec = torch.clamp(((torch.atan2(uv[:, 1], uv[:, 0]) / (2.0 * math.pi) + 0.5) * sectors).long(), max=sectors - 1)
        return (ring * sectors + sec).int()
    s = int(round(math.sqrt(d)))
    rank = torch.empty(m, dtype=torch.int64, device=DEV)
    rank[torch.argsort(uv[:, 0], stable=True)] = torch.arange(m, device=DEV)
    strip = rank * s // m
    inside = torch.argsort(strip * 8.0 + uv[:, 1], stable=True)      # |v| <= pi < 4
    rank[inside] = torch.arange(m, device=DEV)
    first = -(-strip * m // s)
    count = -(-(strip + 1) * m // s) - first
    return (strip * s + (rank - first) * s // count).int()


def _sky(case, seed):
    """Blobs (amplitude, centre x and y, width) and points of a sky, in pixels from the centre."""
    g, nx, ny = _gen(seed, 2), case["nx"], case["ny"]
    u = torch.rand(30, 4, generator=g, device=DEV, dtype=torch.float64)
    sd = (1.0 + 3.0 * u[:20, 3]) * max(nx, ny) / 64.0
    return u[:, 0], (u[:, 1] * nx).floor() - nx // 2, (u[:, 2] * ny).floor() - ny // 2, sd


def _image(case, seed):
    amp, cx, cy, sd = _sky(case, seed)
    xx = torch.arange(case["nx"], device=DEV, dtype=torch.float64) - case["nx"] // 2
    yy = torch.arange(case["ny"], device=DEV, dtype=torch.float64) - case["ny"] // 2
    ex = torch.exp(-(xx[None] - cx[:20, None]) ** 2 / (2.0 * sd[:, None] ** 2))
    ey = torch.exp(-(yy[None] - cy[:20, None]) ** 2 / (2.0 * sd[:, None] ** 2))
    img = torch.einsum("k,ky,kx->yx", amp[:20], ey, ex)
    img[(cy[20:] + case["ny"] // 2).long(), (cx[20:] + case["nx"] // 2).long()] += amp[20:]
    return img


def _measure(case, seed, uv):
    """Noisy visibilities of the sky in closed form, and the noise's standard deviation."""
    amp, cx, cy, sd = _sky(case, seed)
    y = torch.zeros(uv.shape[0], dtype=torch.complex128, device=DEV)
    for k in range(30):
        a = amp[k] * torch.ones((), dtype=torch.float64, device=DEV).expand(uv.shape[0])
        if k < 20:
            a = a * 2.0 * math.pi * sd[k] ** 2 * torch.exp(-0.5 * sd[k] ** 2 * (uv ** 2).sum(dim=1))
        y += torch.polar(a.contiguous(), -(uv[:, 0] * cx[k] + uv[:, 1] * cy[k]))
    sn = (y.abs().square().mean().sqrt() * 10.0 ** (-30.0 / 20.0)).item()
    n = torch.randn(uv.shape[0], 2, generator=_gen(seed, 3), device=DEV, dtype=torch.float64)
    return y + torch.view_as_complex(n) * (sn / math.sqrt(2.0)), sn


def _eps(blocks, nblocks, sn):
    """Bounds at the 99th percentile of the noise: sn / sqrt(2) * sqrt(chi2_0.99(2 M_i)) (Wilson-Hilferty)."""
    k = 2.0 * np.maximum(np.bincount(blocks, minlength=nblocks), 1)
    h = 2.0 / (9.0 * k)
    return sn / math.sqrt(2.0) * np.sqrt(k * (1.0 - h + 2.3263478740408408 * np.sqrt(h)) ** 3)


def _norm2(case, uv):
    """An upper estimate of ||Phi||^2 from the densest part of the coverage: points per
    (2 pi / nx) x (2 pi / ny) cell, averaged over 4 x 4 cells, times the pixels."""
    nx, ny = case["nx"] // 4, case["ny"] // 4
    ix = torch.clamp(((uv[:, 0] / (2.0 * math.pi) + 0.5) * nx).long(), max=nx - 1)
    iy = torch.clamp(((uv[:, 1] / (2.0 * math.pi) + 0.5) * ny).long(), max=ny - 1)
    most = torch.bincount(iy * nx + ix, minlength=nx * ny).max().item()
    return 1.5 * max(most / 16.0, 0.25) * case["nx"] * case["ny"]


def _dde(case, seed):
    d = case["dde"]
    k = 0.1 * torch.randn(case["m"], d, d, 2, generator=_gen(seed, 4), device=DEV, dtype=torch.float64)
    k[:, d // 2, d // 2, 0] += 1.0
    return torch.view_as_complex(k)


def _inputs(case, seed):
    """Everything that a pass reads, on the GPU, and the numbers that go with it."""
    rdt, cdt = (torch.float64, torch.complex128) if case["precision"] == "f64" else (torch.float32, torch.complex64)
    nx, ny = case["nx"], case["ny"]
    if case["kind"] == "psi":
        noise = torch.randn(case["bases"], ny, nx, generator=_gen(seed, 5), device=DEV, dtype=rdt)
        return dict(x=_image(case, seed).to(rdt), coeffs=noise)
    uv = _uv(case, seed)
    if case["kind"] == "phi":
        b = case["batch"]
        x = torch.stack([_image(case, 7919 * seed + k) for k in range(max(b, 1))]).to(rdt)
        g = torch.randn(*((b,) if b else ()), case["m"], 2, generator=_gen(seed, 5), device=DEV, dtype=rdt)
        return dict(uv=uv, x=x if b else x[0].contiguous(), g=torch.view_as_complex(g))
    blk = _blocks(case, uv)
    y, sn = _measure(case, seed, uv)
    host = blk.cpu().numpy()
    out = dict(uv=uv, blocks=blk, host_blocks=host, y=y.to(cdt), eps=_eps(host, case["nblocks"], sn),
               step=dict(STEP, varsigma=1.0 / _norm2(case, uv)), seed=int(seed) + 17,
               p_block=np.full(case["nblocks"], case["p"]), p_basis=np.full(case["bases"], case["p"]))
    if case["dde"]:
        out["dde"] = _dde(case, seed)
    if case.get("weights"):
        out["x"] = _image(case, seed).to(rdt)
    if case.get("adaptive"):
        d = case["nblocks"]
        out["adaptive"] = dict(n=d / 4.0, p_min=0.05, p_max=0.5)
    return out


# ------------------------------------------------------------------ what is timed
def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    ids = tuple(range(case["bases"])) if "bases" in case else (0,)
    kw = dict(precision=case["precision"], basis_ids=ids, levels=case.get("levels", 1))
    if case["kind"] == "psi":
        s["ids"] = ids
        if not case["noalloc"]:
            s["plan"] = Plan(case["nx"], case["ny"], np.zeros((1, 2)), np.zeros(1, np.int32), 1, **kw)
        else:
            s["out"] = torch.empty_like(s["coeffs"])
            psi_adj_noalloc(s["x"], ids, case["levels"], s["out"])      # the one-time set-up
        return s
    kw["kernel_width"] = case["width"]
    uv = s.pop("uv").cpu().numpy()
    if case["kind"] == "phi":
        s["plan"] = Plan(case["nx"], case["ny"], uv, np.zeros(len(uv), np.int32), 1, **kw)
        s["x"].requires_grad_(True)
        return s
    s.pop("blocks")
    if case["csr"]:
        kw["g_mode"] = "csr"
    if case["dde"]:
        kw["dde_kernels"] = s.pop("dde").cpu().numpy()
    s["plan"] = Plan(case["nx"], case["ny"], uv, s.pop("host_blocks"), case["nblocks"], **kw)
    s["state"] = State(s["plan"])
    if case.get("weights"):
        s["w"] = torch.empty(case["bases"], case["ny"], case["nx"], dtype=s["x"].dtype, device=DEV)
    return s


def run(s):
    case, plan = s["case"], s.get("plan")
    if case["kind"] == "phi":
        y = autograd.phi(s["x"], plan)
        (grad,) = torch.autograd.grad(y, s["x"], s["g"])
        return {"y": y.detach(), "grad": grad}
    if case["kind"] == "psi":
        if case["noalloc"]:
            return {"coeffs": psi_adj_noalloc(s["x"], s["ids"], case["levels"], s["out"])}
        return {"coeffs": plan.pd_apply_psi_adj(s["x"]), "image": plan.pd_apply_psi(s["coeffs"])}
    st = s["state"]
    w = plan.pd_sara_weights(s["x"], 0.01, s["w"]) if case.get("weights") else None
    st.pd_state_set_data(s["y"], s["eps"])
    if case["kind"] == "synth":
        st.pd_synthesis_iterate(case["iters"], seed=s["seed"], p_block=s["p_block"], **s["step"])
    else:
        st.pd_iterate(case["iters"], seed=s["seed"], p_block=s["p_block"], p_basis=s["p_basis"],
                      adaptive=s.get("adaptive"), use_graph=case["graph"], weights=w, **s["step"])
    out = {"x": st.x(), "s": st.s(), "v": st.v()}
    if w is not None:
        out["weights"] = w
    return out


# ------------------------------------------------------------------ what it cannot do without
def work(case):
    """Bytes and operations of one pass: per application of Phi or Phi^H the points (two
    coordinates), the visibilities and the image once, 4 J^2 operations a point and the two
    FFTs; per basis the coefficients once, 4 taps per tap pair and pixel over the levels."""
    r = 8 if case["precision"] == "f64" else 4
    n = case["nx"] * case["ny"]
    taps = sum(2 * k for k in range(case.get("bases", 1)))
    wave = 2 * 2 * 2 * taps * n * 4 / 3                       # both passes, both filters, all levels
    if case["kind"] == "psi":
        b = case["bases"]
        both = 1 if case["noalloc"] else 2
        return {"bytes": both * r * n * (1 + b), "flops": both * wave}
    m = case["m"]
    fft = 5 * 2 * n * math.log2(4 * n)                        # the half spectrum of the padded real image
    foot = case["width"] + max(case.get("dde", 0) - 1, 0)
    g = 4 * foot ** 2 * (2 if case.get("dde") else 1)
    if case["kind"] == "phi":
        b = max(case["batch"], 1)
        return {"bytes": 2 * (b * r * (n + 2 * m) + 2 * r * m), "flops": 2 * b * (fft + g * m)}
    p = 0.25 if case.get("adaptive") else case["p"]
    q = case["p"] if case["kind"] == "pd" else 1.0
    b, it = case["bases"], case["iters"]
    entries = foot ** 2 * (4 + (2 if case.get("dde") else 1) * r) if case["csr"] else 2 * r
    per = p * m * (2 * entries + 2 * r * 3) + q * b * n * 2 * r + 4 * n * r
    if case.get("weights"):
        per += q * b * n * r
    ops = 2 * (fft + p * g * m) + q * 2 * wave
    ends = r * (4 * m + 2 * n * (1 + b))                       # the measurements in, the state out
    return {"bytes": it * per + ends, "flops": it * ops}


# ------------------------------------------------------------------ the same in 64 bits, from the definitions
class _Phi:
    """Phi = G F Z with a Kaiser-Bessel kernel on the twice oversampled grid, in 64 bits."""

    def __init__(self, case, uv, dde=None):
        self.nx, self.ny, self.J, self.dde = case["nx"], case["ny"], case["width"], dde
        self.kx, self.ky = 2 * self.nx, 2 * self.ny
        self.beta = math.pi * math.sqrt((self.J / 2.0) ** 2 * 2.25 - 0.8)
        self.c = self._deapodise(self.ny)[:, None] * self._deapodise(self.nx)[None, :]
        self.gx, self.gy = uv[:, 0] * (self.kx / (2.0 * math.pi)), uv[:, 1] * (self.ky / (2.0 * math.pi))

    def _deapodise(self, n):
        xi = (torch.arange(n, device=DEV, dtype=torch.float64) - n / 2) / (2 * n)
        z = torch.sqrt(torch.complex(self.beta ** 2 - (math.pi * self.J * xi) ** 2, torch.zeros_like(xi)))
        return (z / torch.sinh(z)).real / self.J

    def _weights(self, t):
        q = 1.0 - (2.0 * t / self.J) ** 2
        return torch.where(q >= 0, torch.special.i0(self.beta * torch.sqrt(torch.clamp(q, min=0.0))), torch.zeros_like(q))

    def spectrum(self, x):
        z = torch.zeros(self.ky, self.kx, dtype=torch.complex128, device=DEV)
        z[: self.ny, : self.nx] = x.double() * self.c
        return torch.fft.fft2(torch.roll(z, (-(self.ny // 2), -(self.nx // 2)), (0, 1)))

    def crop(self, grid):
        z = torch.fft.ifft2(grid, norm="forward").real
        return torch.roll(z, (self.ny // 2, self.nx // 2), (0, 1))[: self.ny, : self.nx] * self.c

    def _rows(self, at, chunk=1 << 20):
        """For chunks of the points `at`: their places, each footprint cell's index and its weight."""
        ex = 0 if self.dde is None else self.dde.shape[1] - 1
        for k in range(0, at.shape[0], chunk):
            part = at[k:k + chunk]
            gx, gy = self.gx[part], self.gy[part]
            bx, by = torch.floor(gx) - (self.J // 2 - 1), torch.floor(gy) - (self.J // 2 - 1)
            wx = [self._weights(gx - bx - a) for a in range(self.J)]
            wy = [self._weights(gy - by - b) for b in range(self.J)]
            for b in range(self.J + ex):
                ky = (by.long() + b - ex // 2) % self.ky
                for a in range(self.J + ex):
                    kx = (bx.long() + a - ex // 2) % self.kx
                    if self.dde is None:
                        w = wy[b] * wx[a]
                    else:
                        w = sum(wy[b - i] * wx[a - j] * self.dde[part, i, j] for i in range(ex + 1)
                                for j in range(ex + 1) if 0 <= b - i < self.J and 0 <= a - j < self.J)
                    yield k, part.shape[0], ky * self.kx + kx, w

    def degrid(self, grid, at):
        out = torch.zeros(at.shape[0], dtype=torch.complex128, device=DEV)
        flat = grid.reshape(-1)
        for k, n, cell, w in self._rows(at):
            out[k:k + n] += w * flat[cell]
        return out

    def grid(self, v, at, into=None):
        out = torch.zeros(self.ky * self.kx, 2, dtype=torch.float64, device=DEV) if into is None else into
        for k, n, cell, w in self._rows(at):
            out.index_add_(0, cell, torch.view_as_real((w.conj() if w.is_complex() else w) * v[k:k + n]))
        return out

    def back(self, grid):
        return self.crop(torch.view_as_complex(grid).reshape(self.ky, self.kx))


def _daubechies(p):
    y = np.roots([math.comb(p - 1 + k, k) for k in range(p)][::-1])
    c = 1.0 - 2.0 * y
    z = c + np.sqrt(c * c - 1.0 + 0j)
    z = np.where(np.abs(z) < 1.0, z, 1.0 / z)
    h = np.real(np.poly(np.concatenate([-np.ones(p), z])))
    return h * (math.sqrt(2.0) / h.sum())


def _split(x, h, axis):
    """One periodic analysis level along `axis` (low half, then high half)."""
    m, k = x.shape[axis], len(h)
    lo = hi = 0.0
    for j in range(k):
        at = (2 * torch.arange(m // 2, device=DEV) + j) % m
        xs = x.index_select(axis, at)
        lo, hi = lo + h[j] * xs, hi + (-1) ** j * h[k - 1 - j] * xs
    return torch.cat([lo, hi], dim=axis)


def _merge(c, h, axis):
    m, k = c.shape[axis], len(h)
    lo, hi = c.narrow(axis, 0, m // 2), c.narrow(axis, m // 2, m // 2)
    out = torch.zeros_like(c)
    for j in range(k):
        at = (2 * torch.arange(m // 2, device=DEV) + j) % m
        out.index_add_(axis, at, h[j] * lo + (-1) ** j * h[k - 1 - j] * hi)
    return out


def _analysis(x, case, which=None):
    out = []
    for j in range(case["bases"]) if which is None else which:
        c = x.double().clone()
        for lev in range(case["levels"] if j else 0):
            sub = c[: case["ny"] >> lev, : case["nx"] >> lev]
            sub.copy_(_split(_split(sub, _daubechies(j), 1), _daubechies(j), 0))
        out.append(c)
    return torch.stack(out) / math.sqrt(case["bases"])


def _synthesis(s, case):
    out = torch.zeros(case["ny"], case["nx"], dtype=torch.float64, device=DEV)
    for j in range(case["bases"]):
        c = s[j].double().clone()
        for lev in reversed(range(case["levels"] if j else 0)):
            sub = c[: case["ny"] >> lev, : case["nx"] >> lev]
            sub.copy_(_merge(_merge(sub, _daubechies(j), 0), _daubechies(j), 1))
        out += c
    return out / math.sqrt(case["bases"])


def _philox(seed, t, stream, index):
    """Philox-4x64-10 (Salmon, Moraes, Dror and Shaw 2011): a uniform number in [0, 1)."""
    top, c, k = (1 << 64) - 1, [t, stream, index, 0], [seed, 0]
    for _ in range(10):
        a, b = 0xD2E7470EE14C6C93 * c[0], 0xCA5A826395121157 * c[2]
        c = [(b >> 64) ^ c[1] ^ k[0], b & top, (a >> 64) ^ c[3] ^ k[1], a & top]
        k = [(k[0] + 0x9E3779B97F4A7C15) & top, (k[1] + 0xBB67AE8584CAA73B) & top]
    return (c[0] >> 11) * 2.0 ** -53


def _probabilities(res, eps, n, p_min, p_max):
    c = np.maximum(res - eps, 0.0) ** 2 / eps ** 2
    d = len(c)
    if c.sum() == 0.0:
        return np.full(d, n / d)
    q, cap = (n - d * p_min) * c / c.sum(), p_max - p_min
    lo, hi = 0.0, 0.0 if np.all(q <= cap) else cap
    for _ in range(80):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if np.minimum(q + mid, cap).sum() < n - d * p_min else (lo, mid)
    return p_min + np.minimum(q + hi, cap)


def _iterate(case, s, ref):
    """Algorithm 1 (or its synthesis form) from zero, in 64 bits."""
    st, d, b = s["step"], case["nblocks"], case["bases"]
    shape = (case["ny"], case["nx"])
    zero = torch.zeros(shape, dtype=torch.float64, device=DEV)
    x, xt, u = zero.clone(), zero.clone(), zero.clone()
    c = torch.zeros(b, *shape, dtype=torch.float64, device=DEV)        # s, or alpha
    ct = c.clone()
    y, blk = s["y"].to(torch.complex128), s["blocks"].long()
    v, U = torch.zeros_like(y), torch.zeros(ref.ky * ref.kx, 2, dtype=torch.float64, device=DEV)
    eps = torch.from_numpy(s["eps"]).to(DEV)
    sums = lambda r, at: torch.zeros(d, dtype=torch.float64, device=DEV).index_add_(0, blk[at], r.abs() ** 2).sqrt()  # noqa: E731
    everything = torch.arange(y.shape[0], device=DEV)
    res = sums(y, everything).cpu().numpy()
    out, alpha = {}, st["kappa"]
    if case.get("weights"):
        out["weights"] = 0.01 / (0.01 + _analysis(s["x"], case).abs())
        alpha = alpha * out["weights"]
    for t in range(1, case["iters"] + 1):
        p = _probabilities(res, s["eps"], **s["adaptive"]) if case.get("adaptive") else s["p_block"]
        on = np.array([_philox(s["seed"], t, 0, i) < p[i] for i in range(d)])
        if case["kind"] == "synth":
            xt = _synthesis(ct, case)
        at = torch.nonzero(torch.from_numpy(on).to(DEV)[blk])[:, 0]
        if at.numel():
            gap = ref.degrid(ref.spectrum(xt), at) - y[at]
            r = v[at] + gap
            res = np.where(on, sums(gap, at).cpu().numpy(), res)
            new = r * torch.clamp(1.0 - eps / torch.clamp(sums(r, at), min=1e-300), min=0.0)[blk[at]]
            ref.grid(new - v[at], at, U)
            v[at] = new
        if case["kind"] == "synth":
            u = torch.clamp(u + xt, max=0.0)
            q = c - st["tau"] * _analysis(st["sigma"] * u + st["varsigma"] * ref.back(U), case)
            new = torch.sign(q) * torch.clamp(q.abs() - st["tau"] * st["kappa"], min=0.0)
            c, ct = new, 2.0 * new - c
            continue
        for j in range(b):
            if _philox(s["seed"], t, 1, j) < s["p_basis"][j]:
                a = alpha[j] if case["weights"] else torch.full((), alpha, dtype=torch.float64, device=DEV)
                c[j] = torch.maximum(torch.minimum(c[j] + _analysis(xt, case, [j])[0], a), -a)
        new = torch.clamp(x - st["tau"] * (st["sigma"] * _synthesis(c, case) + st["varsigma"] * ref.back(U)), min=0.0)
        x, xt = new, 2.0 * new - x
    return dict(out, x=_synthesis(c, case) if case["kind"] == "synth" else x, s=c, v=v)


def exact(case, seed):
    s = _inputs(case, seed)
    if case["kind"] == "psi":
        out = {"coeffs": _analysis(s["x"], case)}
        return out if case["noalloc"] else dict(out, image=_synthesis(s["coeffs"], case))
    ref = _Phi(case, s["uv"], s.get("dde"))
    if case["kind"] != "phi":
        return _iterate(case, s, ref)
    at = torch.arange(case["m"], device=DEV)
    xs, gs = (s["x"], s["g"]) if case["batch"] else (s["x"][None], s["g"][None])
    y = torch.stack([ref.degrid(ref.spectrum(x), at) for x in xs])
    grad = torch.stack([ref.back(ref.grid(g.to(torch.complex128), at)) for g in gs])
    return {"y": y, "grad": grad} if case["batch"] else {"y": y[0], "grad": grad[0]}
