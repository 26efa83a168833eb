"""The mixed FGMRES outer loop at the shortest and longest restart lengths: it
converges wherever the FP64 oracle's does within the same allowance of
applications, to a solution within 1e-6 of the oracle's when driven to 1e-10,
and where the oracle's does not (restarts too short), it reports the cap with a
residual no larger than 1.1 times the oracle's (restarted residuals, formed in
FP64, of basis vectors that carry float rounding)."""
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


@pytest.mark.parametrize("m", [1, 2, 9, 31, 32])
def test_mixed_fgmres_restart_lengths(m):
    n, h, tol, B = 64, 1.0 / 64, 1e-10, 2
    k = 0.4 / h
    cap = 64 if m < 9 else 400
    H = ohier.build_hierarchy(n, n, h, k, 0.7)
    b = synth.random_complex((B, n + 1, n + 1), 8) / h**2
    s = hm.Solver(n, n, h, k, 0.7, smoother="jacobi", nu_pre=1, nu_post=1, krylov=m, precision="mixed", batch=B,
                  coarse_nodes=0, max_cycles=cap)
    x, st, cyc, rr = s.solve(torch.from_numpy(b).cuda(), tol=tol)
    s.close()
    opt = ocycle.CycleOptions(1, "jacobi", 1, 1, 4.5)
    conv = []
    for q in range(B):
        ref = okry.fgmres_solve(H, b[q].ravel(), tol, opt, m, max_cycles=cap)
        conv.append(ref.converged)
        if ref.converged:
            assert rr[q] <= tol
            assert abs(cyc[q] - ref.cycles) <= max(2, 0.1 * ref.cycles), (cyc[q], ref.cycles)
            assert pu.rel2(x[q].cpu().numpy(), ref.x) <= 1e-6
        else:
            own = np.linalg.norm(b[q].ravel() - H.A[0] @ ref.x) / np.linalg.norm(b[q])
            assert cyc[q] == cap and rr[q] <= 1.1 * own, (cyc[q], rr[q], own)
    assert st == (hm.MG_OK if all(conv) else hm.MG_EMAXIT)
