"""The complex64 cycles of a small and of a large right-hand side: the GMRES(3)
smoother is homogeneous, so b times a power of two takes the same cycles to the
same solution times that power, as far as the stopping test's own float norm
reaches (squares of about 1e-44 to 1e37 per node at the ends used here).

Every kernel that sums a Gram matrix is in: the fine level's march, column
marches and stored stencils (one right-hand side and several per block), the
node-parallel forms, the cluster, the flattened ragged launches and FGMRES.
The stopping norm is exact to a few per cent of itself at the small end, so a
count may differ by one cycle."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2308_13476_gb300 as hm  # noqa: E402

SCALES = [2.0 ** -66, 2.0 ** -40, 2.0 ** 43]
TOL = 1e-6


def _close(x, ref, scale, cyc, cref):
    assert max(abs(int(a) - int(b)) for a, b in zip(cyc, cref)) <= 1, (cyc, cref)
    # each is within TOL times the operator's condition of the solution: about
    # (8 / h^2) / (2 k) = 850 at 129^2 and kh = 0.6 (the eigenvalues next to
    # zero are damped at about 2 k by the absorbing sides)
    d = torch.linalg.vector_norm(x / scale - ref) / torch.linalg.vector_norm(ref)
    assert d.item() <= 2e-3, d.item()


@pytest.mark.parametrize("kw", [dict(), dict(coarse_nodes=0), dict(kvar=True, coarse_nodes=0),
                                dict(kvar=True, coarse_nodes=0, batch=17), dict(coarse_nodes=0, march=0),
                                dict(cycle="W", kvar=True), dict(abc=2), dict(precision="mixed-ff"),
                                dict(krylov=5), dict(krylov=5, coarse_nodes=0)], ids=str)
def test_scaled_right_hand_side(kw):
    kw = dict(kw)
    n, kvar, B = 128, kw.pop("kvar", False), kw.pop("batch", 1)
    kw.setdefault("precision", "mixed")
    h = 1.0 / n
    k = 0.6 / h
    kk = torch.from_numpy(synth.k_field(synth.chi_smooth(n, n, 2), 0.6 * k, k)).cuda() if kvar else k
    b = torch.from_numpy(synth.random_complex((B, n + 1, n + 1), 7)).cuda() / h**2
    s = hm.Solver(n, n, h, kk, 1 / k, smoother="gmres3", nu_pre=2, nu_post=2, batch=B, max_cycles=100, **kw)
    ref, st, cref, _ = s.solve(b, tol=TOL)
    assert st == hm.MG_OK
    for scale in SCALES:
        x, st, cyc, rr = s.solve(b * scale, tol=TOL)
        assert st == hm.MG_OK, (scale, cyc, rr)
        _close(x, ref, scale, cyc, cref)
    s.close()


@pytest.mark.parametrize("flat", [0, 1])
def test_scaled_right_hand_side_of_one_ragged_problem(flat):
    """Every problem of a batch keeps its own scale."""
    sizes = [(n, n, 1.0 / n, 0.6 * n) for n in (64, 96, 128)]
    s = hm.RaggedSolver(sizes, [1 / q[3] for q in sizes], smoother="gmres3", nu_pre=2, nu_post=2, precision="mixed",
                        flat=flat, max_cycles=100)
    b = [torch.from_numpy(synth.random_complex((q[1] + 1, q[0] + 1), 7)).cuda() / q[2] ** 2 for q in sizes]
    ref, st, cref, _ = s.solve(b, tol=TOL)
    assert st == hm.MG_OK
    scales = [2.0 ** 43, 2.0 ** -66, 2.0 ** -66]
    x, st, cyc, rr = s.solve([v * c for v, c in zip(b, scales)], tol=TOL)
    assert st == hm.MG_OK, (cyc, rr)
    for q in range(len(sizes)):
        _close(x[q], ref[q], scales[q], cyc[q:q + 1], cref[q:q + 1])
    s.close()
