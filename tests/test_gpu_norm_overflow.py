"""The mixed path's stopping test past the range of its float norm: a residual
whose squares exceed the largest float is reported as an infinite relative residual
(diverged), and the right-hand sides beside it are solved to the last bit as if
it were not there."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2308_13476_gb300 as hm  # noqa: E402


@pytest.mark.parametrize("n", [24, 128])
@pytest.mark.parametrize("kvar", [False, True])
def test_overflowing_norm_is_infinite(n, kvar):
    h = 1.0 / n
    k = 0.4 / h
    kk = torch.from_numpy(synth.k_field(synth.chi_smooth(n, n, 2), 0.6 * k, k)).cuda() if kvar else k
    s = hm.Solver(n, n, h, kk, 1 / k, smoother="gmres3", nu_pre=2, nu_post=2, precision="mixed", batch=3)
    b = torch.from_numpy(synth.random_complex((3, n + 1, n + 1), 7)).cuda() / h**2
    ref = s.solve(b, tol=1e-8)[0]
    b[1] *= 1e25                      # finite in float, its squares are not
    x, st, cyc, rr = s.solve(b, tol=1e-8)
    assert st == hm.MG_EDIVERGED
    assert cyc[1] == 0 and np.isposinf(rr[1]), rr
    assert rr[0] <= 1e-8 and rr[2] <= 1e-8
    assert torch.equal(x[0], ref[0]) and torch.equal(x[2], ref[2])
    s.close()
