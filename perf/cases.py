"""Workloads of the multigrid Helmholtz solver, from the smallest call to the
largest batch, through the package's public entry points.

``listed()`` names them, ``draw(rng)`` gives more of the same ranges,
``prepare(case, seed)`` makes a case's inputs and the handle a program keeps
between solves, ``run(state)`` makes one pass and returns its outputs,
``work(case)`` counts the bytes and operations of a pass and
``exact(case, seed)`` solves the same problem in 64 bits by block elimination.

Solves run to relative residual 1e-11 unless a case says otherwise: a user who
differences fields or gradients, or who checks a solution, needs them that
tight, and the cycles of a solve to 1e-6 are the first half of them.
"""
import math

import numpy as np
import torch

import paper_2308_13476_gb300 as hm
from paper_2308_13476_gb300 import autograd as hm_autograd

C128 = torch.complex128


def _solve(name, nx, ny, kh, batch, **kw):
    """A constant-k solve: kh = k h, unit length along the longer side."""
    c = dict(kind="solve", name=name, nx=nx, ny=ny, kh=kh, batch=batch, precision="mixed", smoother="gmres3",
             cycle="V", nu=2, krylov=0, tol=1e-11)
    c.update(kw)
    return c


def listed():
    return [
        # the stopping residual of someone else's iterate: one allocation-free call
        dict(kind="residual_norm", name="residual_norm_257", nx=256, ny=256, kh=0.625),
        # the paper's smallest table entries (h = 2^-6, k = 30): omega-Jacobi V(1,1) with shift 0.7, FP64
        _solve("jacobi_fp64_65", 64, 64, 30 / 64, 1, precision="fp64", smoother="jacobi", nu=1, tol=1e-6),
        # one source on the smallest grid of the k sweep (k = 50, kh = 0.625): launch latency
        _solve("one_81", 80, 80, 0.625, 1),
        # one source, FP64 W(2,2) on the k = 100 grid of the sweep: many visits of the small levels
        _solve("one_wcycle_fp64_161", 160, 160, 0.625, 1, precision="fp64", cycle="W"),
        # one source on the bench grid (k = 300 on 1025^2): an interactive solve
        _solve("one_1025", 1024, 1024, 300 / 1024, 1),
        # the bench workload: 64 sources on 1025^2
        _solve("batch64_1025", 1024, 1024, 300 / 1024, 64),
        # a survey's worth of sources where complex128 cycles are wanted
        _solve("batch8_fp64_513", 512, 512, 150 / 512, 8, precision="fp64"),
        # the float-float outer loop on a rectangle, an odd number of sources
        _solve("batch11_ff_769x577", 768, 576, 0.5, 11, precision="mixed-ff"),
        # the Krylov use of the cycle where the cycle alone diverges: FGMRES(20) around Jacobi V(1,1), shift 0.7
        _solve("batch8_fgmres20_513", 512, 512, 150 / 512, 8, smoother="jacobi", nu=1, krylov=20),
        # the layered velocity model at 20 Hz, one source: variable k, stored Galerkin stencils
        dict(kind="layered", name="layered_1281x449", nx=1280, ny=448, freq=20.0, batch=1, precision="mixed",
             tol=1e-11),
        # one step of an inversion: setup for a new model, 16 forward and 16 adjoint solves and the gradient
        dict(kind="gradient", name="gradient16_513", n=512, batch=16, nrec=256, precision="mixed", tol=1e-11),
        # independent problems of different sizes in one call
        dict(kind="ragged", name="ragged16", problems=16, lo=127, hi=640, size_seed=3, precision="mixed", tol=1e-11),
    ]


def _side(rng, lo, hi, cs, levels):
    """A side c * 2^m in [lo, hi] with c from ``cs``, spread over its logarithm."""
    want = lo * (hi / lo) ** rng.random()
    cand = [c * 2 ** m for c in cs for m in range(levels, 11) if lo <= c * 2 ** m <= hi]
    near = sorted(cand, key=lambda v: abs(math.log(v / want)))[:3]
    return rng.choice(near)


def draw(rng):
    kind = rng.choice(["residual_norm", "one", "one", "batch", "batch", "fp64", "jacobi", "fgmres", "layered",
                       "gradient", "ragged"])
    kh = rng.uniform(0.28, 0.625)
    cs = (4, 5, 6, 7)
    if kind == "residual_norm":
        return dict(kind="residual_norm", nx=int(33 * 30 ** rng.random()), ny=int(33 * 30 ** rng.random()), kh=kh)
    if kind == "one":
        n = _side(rng, 64, 1024, cs, 3)
        return _drawn(n, n, kh, 1, precision=rng.choice(["mixed", "mixed", "mixed-ff"]),
                      cycle=rng.choice("VVW") if n <= 320 else "V")
    if kind == "batch":
        nx = _side(rng, 192, 1024, cs, 4)
        ny = rng.choice([nx, nx, nx // 4 * 3])
        # no more than the largest listed case: its nodes, and its cycles (which grow with k)
        most = max(2, min(64, int(60 * 1024 ** 2 / (nx * ny) * min(1.0, 300 / (kh * nx)))))
        return _drawn(nx, ny, kh, int(2 * (most / 2) ** rng.random()), precision=rng.choice(["mixed", "mixed", "mixed-ff"]))
    if kind == "fp64":
        n = _side(rng, 64, 512, cs, 3)
        b = int(1 * 8 ** rng.random())
        return _drawn(n, n, kh, b, precision="fp64", cycle=rng.choice("VW") if n <= 160 else "V")
    if kind == "jacobi":
        n = _side(rng, 48, 256, cs, 3)
        return _drawn(n, n, min(0.47, rng.uniform(15, 30) / n), int(1 * 8 ** rng.random()), precision="fp64",
                      smoother="jacobi", nu=rng.choice([1, 2]), tol=1e-6)
    if kind == "fgmres":
        n = _side(rng, 96, 512, cs, 3)
        return _drawn(n, n, rng.uniform(0.28, 0.4), int(1 * 8 ** rng.random()), smoother="jacobi", nu=1,
                      krylov=rng.choice([10, 20]))
    if kind == "layered":
        f = rng.choice([10.0, 15.0, 20.0])
        nx, ny = {10.0: (640, 224), 15.0: (960, 320), 20.0: (1280, 448)}[f]
        return dict(kind="layered", nx=nx, ny=ny, freq=f * rng.uniform(0.8, 1.0), batch=rng.choice([1, 1, 2]),
                    precision=rng.choice(["mixed", "mixed", "fp64"] if f == 10.0 else ["mixed"]), tol=1e-11)
    if kind == "gradient":
        return dict(kind="gradient", n=_side(rng, 96, 512, cs, 4), batch=rng.randint(3, 16),
                    nrec=rng.choice([32, 64]), precision="mixed", tol=1e-11)
    return dict(kind="ragged", problems=rng.randint(4, 20), lo=127, hi=rng.choice([320, 512, 640]),
                size_seed=rng.randint(10, 1000), precision="mixed", tol=1e-11)


def _drawn(nx, ny, kh, batch, **kw):
    c = _solve("", nx, ny, kh, batch, **kw)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs


def _rng(case, seed):
    return np.random.default_rng([int(seed), case.get("nx", case.get("n", case.get("problems", 0)))])


def _sources(rng, nx, ny, h, batch):
    """Unit point sources 1/h^2 on interior nodes: one anywhere, several along
    the first interior row below the top, jittered, as in a survey line."""
    b = torch.zeros((batch, ny + 1, nx + 1), dtype=C128, device="cuda")
    for s in range(batch):
        if batch == 1:
            i, j = int(rng.integers(1, nx)), int(rng.integers(1, ny))
        else:
            i, j = int(round((s + rng.random()) / batch * nx)), ny - 1
        b[s, j, min(max(i, 1), nx - 1)] = 1.0 / (h * h)
    return b


def _field(rng, ny, nx):
    """A random field smoothed over 20 nodes, in [-1, 1]."""
    f = rng.standard_normal((ny + 1, nx + 1))
    ky, kx = np.fft.fftfreq(ny + 1)[:, None], np.fft.fftfreq(nx + 1)[None, :]
    f = np.real(np.fft.ifft2(np.fft.fft2(f) * np.exp(-2.0 * (np.pi * 20.0) ** 2 * (kx ** 2 + ky ** 2))))
    return 2.0 * (f - f.min()) / (f.max() - f.min()) - 1.0


def _layered(rng, nx, ny, h):
    """Velocities 1500..5500 m/s in eleven dipping layers, three Gaussian
    anomalies and a normal fault with a 150 m throw."""
    z, x = np.meshgrid(np.arange(ny + 1) * h, np.arange(nx + 1) * h, indexing="ij")
    X, Z = nx * h, ny * h
    depth = np.sort(rng.uniform(0.05, 0.95, 10)) * Z
    dip = np.tan(np.deg2rad(rng.uniform(-8, 8, 10)))
    vel = np.sort(rng.uniform(1500.0, 5500.0, 11))
    vel[0], vel[-1] = 1500.0, 5500.0
    zz = z - 150.0 * (x > rng.uniform(0.3, 0.7) * X + z / math.tan(math.radians(60.0)))
    v = vel[sum((zz > depth[t] + (x - 0.5 * X) * dip[t]).astype(np.int64) for t in range(10))]
    for _ in range(3):
        cx, cz, s = rng.uniform(0.1, 0.9) * X, rng.uniform(0.1, 0.9) * Z, rng.uniform(200.0, 500.0)
        v = v * (1.0 + rng.uniform(-0.15, 0.15) * np.exp(-((x - cx) ** 2 + (z - cz) ** 2) / (2 * s * s)))
    return v


def _ragged_sizes(case):
    rng = np.random.default_rng(case["size_seed"])
    cand = np.array(sorted({c * 2 ** m for c in range(4, 8) for m in range(12)}))
    ns = [int(cand[np.argmin(np.abs(cand - n - 1))]) for n in rng.integers(case["lo"], case["hi"] + 1, case["problems"])]
    return [(n, n, 1.0 / n, 0.625 * n) for n in ns]


def _inputs(case, seed):
    """Everything of a case that is not the library's: grids, wavenumbers, right-hand sides."""
    rng = _rng(case, seed)
    kind = case["kind"]
    if kind == "residual_norm":
        nx, ny = case["nx"], case["ny"]
        h = 1.0 / max(nx, ny)
        z = rng.standard_normal((2, ny + 1, nx + 1, 2))
        z = torch.view_as_complex(torch.from_numpy(z).cuda())
        return dict(nx=nx, ny=ny, h=h, k=case["kh"] / h, x=z[0].contiguous(), b=(z[1] / (h * h)).contiguous())
    if kind == "solve":
        nx, ny = case["nx"], case["ny"]
        h = 1.0 / max(nx, ny)
        k = case["kh"] / h
        beta2 = 0.7 if case["smoother"] == "jacobi" else 1.0 / k
        return dict(nx=nx, ny=ny, h=h, k=k, beta2=beta2, rhs=_sources(rng, nx, ny, h, case["batch"]))
    if kind == "layered":
        nx, ny = case["nx"], case["ny"]
        h = 9600.0 / nx
        k = 2 * np.pi * case["freq"] / _layered(rng, nx, ny, h)
        beta2 = 1.0 / (float(k.max()) * nx * h)
        return dict(nx=nx, ny=ny, h=h, k=torch.from_numpy(k).cuda(), beta2=beta2,
                    rhs=_sources(rng, nx, ny, h, case["batch"]))
    if kind == "gradient":
        n, w = case["n"], 2 * math.pi * 15.0
        h = 0.625 * 1800.0 / w
        m = (1.0 + 0.1 * _field(rng, n, n)) / 2000.0 ** 2
        rec = (n - 1) * (n + 1) + np.round((np.arange(case["nrec"]) + 0.5) / case["nrec"] * n).astype(np.int64)
        rhs, rec = _sources(rng, n, n, h, case["batch"]), torch.from_numpy(rec).cuda()
        # observed traces: the outgoing field (i / 4) H0(k r) of each source in the uniform model
        at = rhs.reshape(len(rhs), -1).abs().argmax(1)
        r = (w * h / 2000.0) * ((at % (n + 1))[:, None] - (rec % (n + 1))[None, :]).abs().clamp(min=0.5).double()
        data = torch.complex(-torch.special.bessel_y0(r), torch.special.bessel_j0(r)) / 4.0
        return dict(nx=n, ny=n, h=h, omega=w, m=torch.from_numpy(m).cuda(), rec=rec, data=data, rhs=rhs)
    sizes = _ragged_sizes(case)
    return dict(sizes=sizes, rhs=[_sources(rng, nx, ny, h, 1)[0] for nx, ny, h, _ in sizes])


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    kind = case["kind"]
    if kind == "residual_norm":
        s["out"] = torch.zeros(2, dtype=torch.float64, device="cuda")
    elif kind == "solve":
        s["solver"] = hm.Solver(s["nx"], s["ny"], s["h"], s["k"], s["beta2"], cycle=case["cycle"],
                                smoother=case["smoother"], nu_pre=case["nu"], nu_post=case["nu"],
                                precision=case["precision"], batch=case["batch"], krylov=case["krylov"])
    elif kind == "layered":
        s["solver"] = hm.Solver(s["nx"], s["ny"], s["h"], s["k"], s["beta2"], smoother="gmres3", nu_pre=2, nu_post=2,
                                precision=case["precision"], batch=case["batch"])
    elif kind == "ragged":
        s["solver"] = hm.RaggedSolver(s["sizes"], [1.0 / k for _, _, _, k in s["sizes"]], smoother="gmres3", nu_pre=2,
                                      nu_post=2, precision=case["precision"])
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "residual_norm":
        hm.mg_residual_norm_static(s["nx"], s["ny"], s["h"], s["k"], s["x"], s["b"], s["out"])
        return s["out"]
    if kind == "gradient":
        m = s["m"].detach().requires_grad_(True)
        loss = hm_autograd.misfit(m, s["rhs"], s["rec"], s["data"], (s["nx"], s["ny"], s["h"], s["omega"]),
                                  tol=case["tol"], smoother="gmres3", nu_pre=2, nu_post=2, precision=case["precision"])
        loss.backward()
        return {"loss": loss.detach(), "grad": m.grad}
    x, status, _, _ = s["solver"].solve(s["rhs"], tol=case["tol"])
    return {"x": x, "status": int(status)}


# ------------------------------------------------------------------- work


def work(case):
    """Bytes: right-hand sides read and solutions written once in complex128,
    with the wavenumber field.  Operations: the smoothing steps of the cycles
    that a solve takes (about 0.09 cycles per unit of k and decade for GMRES(3)
    V(2,2) on the unit square), four operator applications and Gram-Schmidt
    per GMRES(3) step, over all levels; complex arithmetic counted in reals."""
    kind = case["kind"]
    if kind == "residual_norm":
        n = (case["nx"] + 1) * (case["ny"] + 1)
        return {"bytes": 32.0 * n, "flops": 30.0 * n}
    if kind == "ragged":
        parts = [work(_solve("", n, n, 0.625, 1, tol=case["tol"])) for n, _, _, _ in _ragged_sizes(case)]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    if kind == "gradient":
        nodes, solves, k = (case["n"] + 1) ** 2, 2 * case["batch"], 0.6 * case["n"]
        steps, extra = 4.0, 16.0 * nodes
    else:
        nodes, solves = (case["nx"] + 1) * (case["ny"] + 1), case["batch"]
        k = case["kh"] * max(case["nx"], case["ny"]) if kind == "solve" else 30.0 * case["freq"]
        steps, extra = 2.0 * case.get("nu", 2), 8.0 * nodes * (kind == "layered")
    decades = -math.log10(case["tol"])
    if case.get("smoother") == "jacobi":
        cycles, step = (0.1 * k * decades if case["krylov"] else 4.0 * k), 20.0 + 10.0 * case["krylov"]
    else:
        cycles, step = (10.0 + 0.02 * k * decades), 150.0
    return {"bytes": 32.0 * nodes * solves + extra, "flops": cycles * steps * step * nodes * solves * 4.0 / 3.0}


# ---------------------------------------------------------- 64-bit reference


def _weights(n):
    w = torch.ones(n + 1, dtype=torch.float64, device="cuda")
    w[0] = w[-1] = 0.5
    return w


def _diagonal(nx, ny, h, k):
    """Diagonal of the row-scaled five-point operator with first-order absorbing rows."""
    wx, wy = _weights(nx)[None, :], _weights(ny)[:, None]
    out = 2.0 * (wx < 1).double() + 2.0 * (wy < 1).double()   # ghost terms 2 i k / h per side
    kk = torch.as_tensor(k, dtype=torch.float64, device="cuda") * torch.ones_like(wx * wy)
    return torch.complex(wx * wy * (4.0 / (h * h) - kk * kk), -wx * wy * out * kk / h)


def _apply(nx, ny, h, diag, u):
    """A u for u of shape (..., ny+1, nx+1)."""
    wx, wy = _weights(nx), _weights(ny)
    y = diag * u
    fx, fy = wy[:, None] / (h * h), wx[None, :] / (h * h)
    y[..., :, 1:] -= fx * u[..., :, :-1]
    y[..., :, :-1] -= fx * u[..., :, 1:]
    y[..., 1:, :] -= fy * u[..., :-1, :]
    y[..., :-1, :] -= fy * u[..., 1:, :]
    return y


class _Direct:
    """Block elimination of the five-point matrix along the longer side."""

    def __init__(self, nx, ny, h, k):
        self.a = (nx, ny, h)
        self.diag = _diagonal(nx, ny, h, k)
        self.turn = nx > ny
        d = self.diag.T if self.turn else self.diag
        n, lines = d.shape[1] - 1, d.shape[0]
        across = _weights(lines - 1)
        self.c = (-_weights(n) / (h * h)).to(C128)[:, None]
        off = torch.diag(torch.ones(n, dtype=C128, device="cuda"), 1)
        off = -(off + off.T) / (h * h)
        self.inv = []
        for j in range(lines):
            s = torch.diag(d[j]) + across[j] * off
            if j:
                s = s - self.c * self.inv[-1] * self.c.T
            self.inv.append(torch.linalg.inv(s))

    def _once(self, b):
        b = b.transpose(-1, -2) if self.turn else b
        z = [b[:, 0, :].T]
        for j in range(1, b.shape[1]):
            z.append(b[:, j, :].T - self.c * (self.inv[j - 1] @ z[-1]))
        u = [self.inv[-1] @ z[-1]]
        for j in range(b.shape[1] - 2, -1, -1):
            u.append(self.inv[j] @ (z[j] - self.c * u[-1]))
        u = torch.stack(u[::-1]).permute(2, 0, 1)
        return u.transpose(-1, -2).contiguous() if self.turn else u.contiguous()

    def __call__(self, b):
        u = self._once(b)
        for _ in range(2):
            u = u + self._once(b - _apply(*self.a, self.diag, u))
        return u


def _direct(nx, ny, h, k):
    """The direct solver, or None where it would take too long."""
    return _Direct(nx, ny, h, k) if min(nx, ny) <= 640 else None


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "residual_norm":
        d = _diagonal(s["nx"], s["ny"], s["h"], s["k"])
        r = s["b"] - _apply(s["nx"], s["ny"], s["h"], d, s["x"])
        return torch.stack([torch.linalg.vector_norm(r), torch.linalg.vector_norm(s["b"])])
    if kind == "ragged":
        found = {}
        for n, _, h, k in set(s["sizes"]):
            a = _direct(n, n, h, k) if n <= 512 else None
            found[n] = a and {i: a(b[None])[0] for i, b in enumerate(s["rhs"]) if s["sizes"][i][0] == n}
        return {"x": [found[n] and found[n][i] for i, (n, _, _, _) in enumerate(s["sizes"])], "status": None}
    if kind == "gradient":
        nx, ny, h, w, m = s["nx"], s["ny"], s["h"], s["omega"], s["m"]
        a = _direct(nx, ny, h, w * torch.sqrt(m))
        u = a(s["rhs"])
        res = u.reshape(len(u), -1)[:, s["rec"]] - s["data"]
        g = torch.zeros_like(u).reshape(len(u), -1)
        g[:, s["rec"]] = res
        lam = a(g.reshape(u.shape).conj()).conj()
        wx, wy = _weights(nx)[None, :], _weights(ny)[:, None]
        out = 2.0 * (wx < 1).double() + 2.0 * (wy < 1).double()
        dd = torch.complex(-wx * wy * w * w * torch.ones_like(m), -wx * wy * out / h * w / (2.0 * torch.sqrt(m)))
        return {"loss": 0.5 * (res.abs() ** 2).sum(), "grad": -(lam.conj() * dd * u).sum(0).real}
    a = _direct(s["nx"], s["ny"], s["h"], s["k"])
    return a and {"x": a(s["rhs"]), "status": None}
