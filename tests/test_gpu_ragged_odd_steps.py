"""Flattened ragged batches (flat = 1) in the mixed path with odd and zero numbers
of smoothing steps, where the fine level's iterate ends in its second vector,
and W-cycles, with problems whose whole cycle is one cluster launch beside
problems with grid-wide levels: each problem takes the cycles of its own solve,
and its solution is that solve's.

Both run the same complex64 arithmetic but for where sums are cut into blocks,
so the solutions, driven to 1e-10, agree to the mixed path's 1e-6 and the
counts within 10 % (at least two)."""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2308_13476_gb300 as hm  # noqa: E402


@pytest.mark.parametrize("nu", [(1, 2), (3, 0), (0, 1), (2, 1)])
@pytest.mark.parametrize("cycle", ["V", "W"])
@pytest.mark.parametrize("coarse_nodes", [1100, 40])
def test_each_problem_equals_its_own_solve(nu, cycle, coarse_nodes):
    sizes = [(nx, ny, 1.0 / max(nx, ny), 0.4 * max(nx, ny)) for nx, ny in ((40, 24), (160, 160), (96, 64), (320, 192))]
    kw = dict(smoother="gmres3", nu_pre=nu[0], nu_post=nu[1], cycle=cycle, precision="mixed", coarse_nodes=coarse_nodes)
    b = [torch.from_numpy(synth.random_complex((q[1] + 1, q[0] + 1), 3)).cuda() / q[2] ** 2 for q in sizes]
    s = hm.RaggedSolver(sizes, [1 / q[3] for q in sizes], flat=1, **kw)
    x, st, cyc, rr = s.solve(b, tol=1e-10)
    assert st == hm.MG_OK
    s.close()
    for q, (nx, ny, h, k) in enumerate(sizes):
        own = hm.Solver(nx, ny, h, k, 1 / k, **kw)
        xo, st, co, _ = own.solve(b[q][None], tol=1e-10)
        own.close()
        assert st == hm.MG_OK
        assert abs(cyc[q] - co[0]) <= max(2, 0.1 * co[0]), (q, cyc[q], co)
        assert (torch.linalg.vector_norm(x[q] - xo[0]) / torch.linalg.vector_norm(xo)).item() <= 1e-6, q
