"""The small levels of the coarse-cycle launch in the mixed path: the zero iterate
of the first sweep, transfers between levels held by a few rows of many blocks
and by two or three blocks, stored stencils on chip and partly on chip, and
W-cycles, whose later visits start from a non-zero iterate.

Each solve, driven to 1e-10, takes the FP64 oracle's cycles to 10 % (at least
two) and its solution agrees to the mixed path's 1e-6; one FP64 cycle of the
same hierarchies to 1e-10 node by node."""
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

# fine grids of 153 nodes and more; coarsest grids of 9, 16, 9, 36, 6, 20, 36 and 6 nodes
GRIDS = [(16, 16), (24, 24), (32, 32), (80, 80), (32, 64), (72, 8), (8, 136), (8, 16)]
CYCLES = [("jacobi", "V", (1, 1)), ("jacobi", "W", (2, 1)), ("jacobi", "W", (0, 1)), ("gmres3", "W", (1, 1)),
          ("gmres3", "V", (2, 1))]


def _problem(nx, ny, kvar, smoother):
    h = 1.0 / max(nx, ny)
    k = (0.2 if smoother == "jacobi" else 0.4) / h
    beta2 = 0.7 if smoother == "jacobi" else 1 / k
    return h, synth.k_field(synth.chi_smooth(nx, ny, 3), 0.6 * k, k) if kvar else k, beta2


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("nx,ny", GRIDS)
@pytest.mark.parametrize("kvar", [False, True])
@pytest.mark.parametrize("smoother,cycle,nu", CYCLES)
def test_mixed_solve(nx, ny, kvar, smoother, cycle, nu):
    h, k, beta2 = _problem(nx, ny, kvar, smoother)
    H = ohier.build_hierarchy(nx, ny, h, k, beta2)
    opt = ocycle.CycleOptions({"V": 1, "W": 2}[cycle], smoother, nu[0], nu[1], 4.5)
    for B in (1, 5):
        b = synth.random_complex((B, ny + 1, nx + 1), 5) / h**2
        s = hm.Solver(nx, ny, h, _dev(k) if kvar else k, beta2, cycle=cycle, smoother=smoother, nu_pre=nu[0],
                      nu_post=nu[1], precision="mixed", batch=B, max_cycles=600)
        x, st, cyc, rr = s.solve(_dev(b), tol=1e-10)
        s.close()
        assert st == hm.MG_OK
        for q in {0, B - 1}:
            ref = ocycle.mg_solve(H, b[q].ravel(), 1e-10, opt, max_cycles=600)
            assert ref.converged
            assert abs(cyc[q] - ref.cycles) <= max(2, 0.1 * ref.cycles), (B, cyc[q], ref.cycles)
            assert pu.rel2(x[q].cpu().numpy(), ref.x) <= 1e-6, B


@pytest.mark.parametrize("nx,ny", GRIDS)
@pytest.mark.parametrize("smoother,cycle,nu", CYCLES)
def test_one_fp64_cycle_with_stored_stencils(nx, ny, smoother, cycle, nu):
    h, k, beta2 = _problem(nx, ny, True, smoother)
    H = ohier.build_hierarchy(nx, ny, h, k, beta2)
    opt = ocycle.CycleOptions({"V": 1, "W": 2}[cycle], smoother, nu[0], nu[1], 4.5)
    b = synth.random_complex((ny + 1, nx + 1), 5) / h**2
    x0 = synth.random_complex((ny + 1, nx + 1), 6)
    s = hm.Solver(nx, ny, h, _dev(k), beta2, cycle=cycle, smoother=smoother, nu_pre=nu[0], nu_post=nu[1], max_cycles=1)
    x, st, cyc, rr = s.solve(_dev(b), x=_dev(x0)[None], tol=1e-300)
    s.close()
    ref = ocycle.mg_cycle(H, 0, x0.ravel(), b.ravel(), opt).reshape(ny + 1, nx + 1)
    pu.assert_close(x[0].cpu().numpy(), ref, 1e-10, (ny + 1, nx + 1), "one cycle")
