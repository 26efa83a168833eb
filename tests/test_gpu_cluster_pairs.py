"""The coarse-cycle launch of a batch of about 64 right-hand sides, whose
clusters have two blocks (a device of about 150 SMs runs at most 38 clusters of
four and 76 of two at once): the smallest exchange, in which the sums of a
cluster are fewer than a warp's lanes.

One FP64 cycle is held to the 1e-10 node-by-node bar of the other execution
modes, a mixed solve driven to 1e-10 to 1e-6 of the FP64 solution."""
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


@pytest.mark.parametrize("nx,ny", [(64, 32), (32, 64), (20, 12)])
@pytest.mark.parametrize("B", [41, 64, 76])
@pytest.mark.parametrize("smoother,cycle,nu", [("gmres3", "V", (2, 1)), ("jacobi", "W", (1, 2))])
def test_one_fp64_cycle_of_clusters_of_two(nx, ny, B, smoother, cycle, nu):
    h = 1.0 / max(nx, ny)
    k, beta2 = 0.4 / h, 0.1
    H = ohier.build_hierarchy(nx, ny, h, k, beta2)
    opt = ocycle.CycleOptions({"V": 1, "W": 2}[cycle], smoother, nu[0], nu[1], 4.5)
    b = synth.random_complex((B, ny + 1, nx + 1), 5) / h**2
    x0 = synth.random_complex((B, ny + 1, nx + 1), 6)
    s = hm.Solver(nx, ny, h, k, beta2, cycle=cycle, smoother=smoother, nu_pre=nu[0], nu_post=nu[1], max_cycles=1,
                  batch=B)
    x, st, cyc, rr = s.solve(_dev(b), x=_dev(x0), tol=1e-300)
    assert st == hm.MG_EMAXIT
    for q in (0, B // 2, B - 1):
        ref = ocycle.mg_cycle(H, 0, x0[q].ravel(), b[q].ravel(), opt).reshape(ny + 1, nx + 1)
        pu.assert_close(x[q].cpu().numpy(), ref, 1e-10, (ny + 1, nx + 1), f"rhs {q}")
    s.close()


@pytest.mark.parametrize("nx,ny", [(64, 32), (96, 96)])
def test_mixed_solve_of_clusters_of_two(nx, ny):
    B, h = 64, 1.0 / max(nx, ny)
    k = 0.6 / h
    b = synth.random_complex((B, ny + 1, nx + 1), 7) / h**2
    H = ohier.build_hierarchy(nx, ny, h, k, 1 / k)
    s = hm.Solver(nx, ny, h, k, 1 / k, smoother="gmres3", nu_pre=2, nu_post=2, precision="mixed", batch=B)
    x, st, cyc, rr = s.solve(_dev(b), tol=1e-10)
    assert st == hm.MG_OK
    for q in (0, B - 1):
        ref = ocycle.mg_solve(H, b[q].ravel(), 1e-12, ocycle.CycleOptions(1, "gmres3", 2, 2, 4.5))
        assert pu.rel2(x[q].cpu().numpy(), ref.x) <= 1e-6
    s.close()
