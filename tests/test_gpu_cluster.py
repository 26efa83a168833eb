"""The coarse-cycle cluster launch against the oracle at the sizes where its
slabs can go wrong: fewer rows than blocks, last slabs of one and two rows,
wide and tall grids, a level of one slab, every cluster size that a batch
gives, and all operator kinds (fine level, Kronecker form, stored stencils).

One FP64 cycle from a random iterate is held to the 1e-10 node-by-node bar of
the other execution modes; a mixed solve driven to 1e-10 to the mixed path's
1e-6 of the FP64 solution.
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

# nx, ny, variable k: 33 + 1 rows over 16 blocks (last slab short), wide and
# tall grids, coarsest grids of 9, 30 and 198 nodes
GRIDS = [(32, 32, False), (96, 16, False), (16, 112, False), (40, 24, True), (84, 32, True), (12, 12, False)]


def _problem(nx, ny, kvar, seed):
    h = 1.0 / max(nx, ny)
    k = 0.4 / h
    if kvar:
        k = synth.k_field(synth.chi_smooth(nx, ny, seed), 0.6 * k, k)
    return h, k


def _dev(a, dtype=torch.complex128):
    return torch.from_numpy(np.ascontiguousarray(a)).to(dtype=dtype, device="cuda")


@pytest.mark.parametrize("nx,ny,kvar", GRIDS)
@pytest.mark.parametrize("smoother,cycle,nu,abc", [("gmres3", "V", (2, 1), 1), ("jacobi", "W", (1, 2), 1),
                                                   ("gmres3", "W", (0, 1), 2)])
def test_one_fp64_cycle_matches_oracle(nx, ny, kvar, smoother, cycle, nu, abc):
    h, k = _problem(nx, ny, kvar, 3)
    beta2 = 0.1
    H = ohier.build_hierarchy(nx, ny, h, k, beta2, abc=abc)
    opt = ocycle.CycleOptions({"V": 1, "W": 2}[cycle], smoother, nu[0], nu[1], 4.5)
    for B in (1, 3):
        b = synth.random_complex((B, ny + 1, nx + 1), 5) / h**2
        x0 = synth.random_complex((B, ny + 1, nx + 1), 6)
        for cn in (1100, 40):   # the whole cycle in the cluster, and its small levels only
            s = hm.Solver(nx, ny, h, _dev(k, torch.float64) if kvar else k, beta2, cycle=cycle, smoother=smoother,
                          nu_pre=nu[0], nu_post=nu[1], max_cycles=1, batch=B, coarse_nodes=cn, abc=abc)
            x, st, cyc, rr = s.solve(_dev(b), x=_dev(x0), tol=1e-300)
            assert st == hm.MG_EMAXIT
            for q in range(B):
                ref = ocycle.mg_cycle(H, 0, x0[q].ravel(), b[q].ravel(), opt).reshape(ny + 1, nx + 1)
                pu.assert_close(x[q].cpu().numpy(), ref, 1e-10, (ny + 1, nx + 1), f"rhs {q}, coarse_nodes {cn}")
            s.close()


@pytest.mark.parametrize("nx,ny,B", [(64, 64, 1), (64, 64, 12), (48, 80, 20), (32, 32, 90)])
def test_mixed_solve_on_every_cluster_size(nx, ny, B):
    h = 1.0 / max(nx, ny)
    k = 0.6 / h
    b = synth.random_complex((B, ny + 1, nx + 1), 7) / h**2
    opt = ocycle.CycleOptions(1, "gmres3", 2, 2, 4.5)
    H = ohier.build_hierarchy(nx, ny, h, k, 1 / k)
    s = hm.Solver(nx, ny, h, k, 1 / k, smoother="gmres3", nu_pre=2, nu_post=2, precision="mixed", batch=B)
    x, st, cyc, rr = s.solve(_dev(b), tol=1e-10)
    assert st == hm.MG_OK
    for q in (0, B - 1):
        ref = ocycle.mg_solve(H, b[q].ravel(), 1e-12, opt)
        assert pu.rel2(x[q].cpu().numpy(), ref.x) <= 1e-6
    s.close()
