"""FP64 refinement residual of the mixed path (row march with diagonal pair
sums) at the sizes where its strips and chunks can go wrong: one strip, strips
of exactly 62 inner columns and one more or less, the fewest rows, several
chunks, variable k, second-order absorbing rows, right-hand sides side by side.

The relative residual of a random iterate, which the solve reports before its
first cycle, against the oracle's matrix: each residual component is rounded to
binary32 once (2^-24 relative), its square and the sums within a warp in
binary32 (at most eight roundings of the square), so the norm is within
5 x 2^-24 = 3e-7 relative; a wrong node of random data changes it by 1e-5 or
more on these grids."""
import numpy as np
import pytest

import synth
from oracle import problem as oprob

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2308_13476_gb300 as hm  # noqa: E402


def _dev(a, dtype=torch.complex128):
    return torch.from_numpy(np.ascontiguousarray(a)).to(dtype=dtype, device="cuda")


@pytest.mark.parametrize("nx,ny", [(6, 6), (62, 8), (64, 6), (124, 12), (126, 60), (128, 200), (186, 40), (500, 16)])
@pytest.mark.parametrize("kvar,abc,B", [(False, 1, 1), (True, 1, 3), (False, 2, 2), (True, 2, 1)])
def test_reported_residual_of_a_random_iterate(nx, ny, kvar, abc, B):
    h = 1.0 / max(nx, ny)
    k = 0.5 / h
    kmax = k
    if kvar:
        k = synth.k_field(synth.chi_smooth(nx, ny, 4), 0.6 * k, k)
    A = oprob.helmholtz_matrix(nx, ny, h, k, abc=abc)
    x0 = synth.random_complex((B, ny + 1, nx + 1), 7)
    b = synth.random_complex((B, ny + 1, nx + 1), 8) / h**2
    s = hm.Solver(nx, ny, h, _dev(k, torch.float64) if kvar else k, 1 / kmax, smoother="gmres3", nu_pre=1, nu_post=1,
                  precision="mixed", batch=B, abc=abc)
    _, st, cyc, rr = s.solve(_dev(b), x=_dev(x0), tol=1e300)
    assert st == hm.MG_OK and list(cyc) == [0] * B
    for q in range(B):
        ref = np.linalg.norm(b[q].ravel() - A @ x0[q].ravel()) / np.linalg.norm(b[q])
        assert abs(rr[q] - ref) <= 3e-7 * ref
    s.close()
