"""Weighted-Jacobi cycles whose coarse levels run as grid-wide kernels: the first
sweep on a zero iterate (no application, the iterate not read or cleared) and
the later ones as column marches on Kronecker-form levels, in both precisions,
with one and several sweeps, W-cycles (second visits start from a non-zero
iterate) and right-hand sides side by side; and the FGMRES outer loop's MGS and
back-substitution chains at the shortest and longest restart lengths.

One FP64 cycle equals the oracle's to 1e-10 node by node, the bar of the other
execution modes; an FGMRES solve takes the oracle's number of applications and
its solution agrees to 1e-9 (64-bit arithmetic in another order over at most 64
preconditioned steps to 1e-6), a mixed one to 1e-6 when driven to 1e-10."""
import numpy as np
import pytest

import parity_util as pu
import synth
from oracle import cycle as ocycle
from oracle import hierarchy as ohier
from oracle import krylov as okry

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2308_13476_gb300 as hm  # noqa: E402


def _dev(a, dtype=torch.complex128):
    return torch.from_numpy(np.ascontiguousarray(a)).to(dtype=dtype, device="cuda")


@pytest.mark.parametrize("nx,ny", [(64, 64), (136, 40), (72, 200)])
@pytest.mark.parametrize("cycle,nu,kvar,B", [("V", (1, 1), False, 1), ("W", (2, 1), False, 3), ("V", (0, 2), False, 2),
                                             ("W", (1, 1), True, 1)])
def test_one_fp64_jacobi_cycle_matches_oracle(nx, ny, cycle, nu, kvar, B):
    h = 1.0 / max(nx, ny)
    k = 0.4 / h
    if kvar:
        k = synth.k_field(synth.chi_smooth(nx, ny, 3), 0.6 * k, k)
    H = ohier.build_hierarchy(nx, ny, h, k, 0.7)
    opt = ocycle.CycleOptions({"V": 1, "W": 2}[cycle], "jacobi", nu[0], nu[1], 4.5)
    b = synth.random_complex((B, ny + 1, nx + 1), 5) / h**2
    x0 = synth.random_complex((B, ny + 1, nx + 1), 6)
    s = hm.Solver(nx, ny, h, _dev(k, torch.float64) if kvar else k, 0.7, cycle=cycle, smoother="jacobi", nu_pre=nu[0],
                  nu_post=nu[1], max_cycles=1, batch=B, coarse_nodes=0)
    x, st, cyc, rr = s.solve(_dev(b), x=_dev(x0), tol=1e-300)
    assert st == hm.MG_EMAXIT
    for q in range(B):
        ref = ocycle.mg_cycle(H, 0, x0[q].ravel(), b[q].ravel(), opt).reshape(ny + 1, nx + 1)
        pu.assert_close(x[q].cpu().numpy(), ref, 1e-10, (ny + 1, nx + 1), f"rhs {q}")
    s.close()


@pytest.mark.parametrize("m", [1, 2, 9, 32])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_fgmres_restart_lengths(m, precision):
    n, h = 64, 1.0 / 64
    k = 0.4 / h
    H = ohier.build_hierarchy(n, n, h, k, 0.7)
    b = synth.random_complex((2, n + 1, n + 1), 8) / h**2
    tol = 1e-6 if precision == "fp64" else 1e-10
    s = hm.Solver(n, n, h, k, 0.7, smoother="jacobi", nu_pre=1, nu_post=1, krylov=m, precision=precision, batch=2,
                  coarse_nodes=0, max_cycles=64 if m < 9 else 400)
    x, st, cyc, rr = s.solve(_dev(b), tol=tol)
    opt = ocycle.CycleOptions(1, "jacobi", 1, 1, 4.5)
    for q in range(2):
        ref = okry.fgmres_solve(H, b[q].ravel(), tol, opt, m, max_cycles=64 if m < 9 else 400)
        if precision == "fp64":
            assert cyc[q] == ref.cycles
            assert pu.rel2(x[q].cpu().numpy(), ref.x) <= 1e-9
        elif st == hm.MG_OK:
            assert ref.converged
            assert pu.rel2(x[q].cpu().numpy(), ref.x) <= 1e-6
    s.close()
