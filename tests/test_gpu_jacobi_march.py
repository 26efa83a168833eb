"""Weighted-Jacobi sweeps of the Kronecker-form levels as column marches and
node-parallel, on both sides of the size at which the automatic rule changes
between them: a forced march (march = 1), none (march = 0) and the rule
(march = -1) take the same sweeps.  FP64 iterates of one cycle agree with the
oracle's to 1e-10 node by node, the bar of the other execution modes; mixed
solves driven to 1e-9 agree with each other to 1e-6."""
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

# level 1 of 33^2, 37 x 69 and 161 x 161 nodes: 1089 to 51842 over the right-hand sides
GRIDS = [(64, 64), (72, 136), (320, 320)]


@pytest.mark.parametrize("nx,ny", GRIDS)
@pytest.mark.parametrize("B", [1, 2])
def test_fp64_cycle_in_every_form(nx, ny, B):
    h = 1.0 / max(nx, ny)
    k = 0.4 / h
    H = ohier.build_hierarchy(nx, ny, h, k, 0.7)
    b = synth.random_complex((B, ny + 1, nx + 1), 5) / h**2
    x0 = synth.random_complex((B, ny + 1, nx + 1), 6)
    ref = [ocycle.mg_cycle(H, 0, x0[q].ravel(), b[q].ravel(), ocycle.CycleOptions(1, "jacobi", 2, 2, 4.5))
           for q in range(B)]
    for march in (-1, 0, 1):
        s = hm.Solver(nx, ny, h, k, 0.7, smoother="jacobi", nu_pre=2, nu_post=2, max_cycles=1, batch=B,
                      coarse_nodes=0, march=march)
        x, st, cyc, rr = s.solve(torch.from_numpy(b).cuda(), x=torch.from_numpy(x0).cuda(), tol=1e-300)
        s.close()
        for q in range(B):
            pu.assert_close(x[q].cpu().numpy(), ref[q].reshape(ny + 1, nx + 1), 1e-10, (ny + 1, nx + 1),
                            f"march {march}, rhs {q}")


@pytest.mark.parametrize("n,B", [(64, 1), (160, 4), (160, 8)])   # level 1: 1089, 26244 and 52488 nodes
def test_mixed_solve_in_every_form(n, B):
    h = 1.0 / n
    k = 0.2 / h
    b = torch.from_numpy(synth.random_complex((B, n + 1, n + 1), 5)).cuda() / h**2
    xs = []
    for march in (-1, 0, 1):
        s = hm.Solver(n, n, h, k, 0.7, smoother="jacobi", nu_pre=1, nu_post=1, krylov=10, precision="mixed", batch=B,
                      coarse_nodes=0, march=march, max_cycles=400)
        x, st, cyc, rr = s.solve(b, tol=1e-9)
        s.close()
        assert st == hm.MG_OK
        xs.append(x)
    for x in xs[1:]:
        assert (torch.linalg.vector_norm(x - xs[0]) / torch.linalg.vector_norm(x)).item() <= 1e-6
