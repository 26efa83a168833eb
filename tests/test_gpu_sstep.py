"""complex64 GMRES(3) smoothing in s-step form at the sizes where its kernels
can go wrong: grids of one strip, strips that end on the last column, a last
strip of one column, fewer rows than the boundary bands, odd and zero numbers
of smoothing steps (the iterate alternates between two vectors), variable k,
second-order absorbing rows, the float-float outer loop and the FGMRES
preconditioner.

The smoother runs inside the mixed path, so each solve is held to that path's
bar: driven to relative residual 1e-10, the solution agrees with the FP64
oracle's to 1e-6, and a wrong smoother would show in the cycle count, which
stays within 10 % (at least two) of the oracle's FP64 count.
"""
import numpy as np
import pytest

import parity_util as pu
import synth
from oracle import cycle as ocycle
from oracle import hierarchy as ohier

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2308_13476_gb300 as hm  # noqa: E402


def _dev(a, dtype=torch.complex128):
    return torch.from_numpy(np.ascontiguousarray(a)).to(dtype=dtype, device="cuda")


@pytest.mark.parametrize("nx,ny", [(6, 6), (54, 16), (56, 8), (110, 24), (112, 40), (64, 6), (168, 168)])
@pytest.mark.parametrize("kw", [dict(), dict(kvar=True, nu=(1, 2), batch=2), dict(abc=2, nu=(2, 1)),
                                dict(precision="mixed-ff", nu=(0, 3)), dict(nu=(3, 0), batch=3),
                                dict(coarse_nodes=40, krylov=5)], ids=str)
def test_mixed_solve_matches_oracle(nx, ny, kw):
    kw = dict(kw)
    kvar, nu, B = kw.pop("kvar", False), kw.pop("nu", (2, 2)), kw.pop("batch", 1)
    kw.setdefault("precision", "mixed")
    kw.setdefault("coarse_nodes", 0)   # every level as grid-wide kernels
    h = 1.0 / max(nx, ny)
    k = 0.4 / h
    kmax = k
    if kvar:
        k = synth.k_field(synth.chi_smooth(nx, ny, 2), 0.6 * k, k)
    b = synth.random_complex((B, ny + 1, nx + 1), 9) / h**2
    H = ohier.build_hierarchy(nx, ny, h, k, 1 / kmax, abc=kw.get("abc", 1))
    opt = ocycle.CycleOptions(1, "gmres3", nu[0], nu[1], 4.5)
    s = hm.Solver(nx, ny, h, _dev(k, torch.float64) if kvar else k, 1 / kmax, smoother="gmres3", nu_pre=nu[0],
                  nu_post=nu[1], batch=B, **kw)
    x, st, cyc, rr = s.solve(_dev(b), tol=1e-10)
    assert st == hm.MG_OK
    for q in (0, B - 1):
        ref = ocycle.mg_solve(H, b[q].ravel(), 1e-10, opt)
        assert ref.converged
        assert pu.rel2(x[q].cpu().numpy(), ref.x) <= 1e-6, q
        if not kw.get("krylov"):
            assert abs(cyc[q] - ref.cycles) <= max(2, 0.1 * ref.cycles), (cyc[q], ref.cycles)
    s.close()


@pytest.mark.parametrize("B", [5, 13, 25])
def test_stored_stencils_share_blocks_between_right_hand_sides(B):
    """Variable k on 257^2: the first coarse level (129^2 stored stencils) runs
    one right-hand side per block in blocks of 512 threads (B = 5), two (13) and
    four (25), the last group of each a partial one; a zero right-hand side
    leaves its group's shared reduction to the others."""
    n, h = 256, 1.0 / 256
    k = synth.k_field(synth.chi_smooth(n, n, 2), 0.24 / h, 0.4 / h)
    kmax = float(k.max())
    b = synth.random_complex((B, n + 1, n + 1), 11) / h**2
    b[2] = 0.0
    H = ohier.build_hierarchy(n, n, h, k, 1 / kmax)
    s = hm.Solver(n, n, h, _dev(k, torch.float64), 1 / kmax, smoother="gmres3", nu_pre=2, nu_post=2, precision="mixed",
                  batch=B)
    x, st, cyc, rr = s.solve(_dev(b), tol=1e-10)
    assert st == hm.MG_OK
    assert cyc[2] == 0 and torch.count_nonzero(x[2]).item() == 0
    ref = ocycle.mg_solve(H, b[B - 1].ravel(), 1e-10, ocycle.CycleOptions(1, "gmres3", 2, 2, 4.5))
    assert pu.rel2(x[B - 1].cpu().numpy(), ref.x) <= 1e-6
    assert abs(cyc[B - 1] - ref.cycles) <= max(2, 0.1 * ref.cycles)
    # the others by their residual with the oracle's matrix
    for q in range(B):
        if q != 2:
            assert pu.rel2(H.A[0] @ x[q].cpu().numpy().ravel(), b[q].ravel()) <= 1.1e-10
    s.close()
