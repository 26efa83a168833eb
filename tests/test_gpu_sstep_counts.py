"""Cycle counts of the complex64 GMRES(3) steps in s-step form against the
complex128 path, whose steps keep the Arnoldi form: constant and variable k, V-
and W-cycles, both transfers, to 1e-6 and to 1e-11.  The least-squares minimum
is flat, so the form of its solution should not show: the counts stay within 10 %
(at least two), the bar of the mixed path's other tests."""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2308_13476_gb300 as hm  # noqa: E402


@pytest.mark.parametrize("n,kh,kw", [(160, 0.625, dict()), (160, 0.625, dict(cycle="W")), (160, 0.4, dict(kvar=True)),
                                     (96, 0.4, dict(kvar=True, cycle="W")), (64, 0.625, dict(transfer="linear")),
                                     (160, 0.625, dict(coarse_nodes=0, nu=1))], ids=str)
@pytest.mark.parametrize("tol", [1e-6, 1e-11])
def test_counts_of_the_s_step_and_the_arnoldi_form(n, kh, kw, tol):
    kw = dict(kw)
    kvar, nu = kw.pop("kvar", False), kw.pop("nu", 2)
    h = 1.0 / n
    k = kh / h
    kk = torch.from_numpy(synth.k_field(synth.chi_smooth(n, n, 2), 0.6 * k, k)).cuda() if kvar else k
    b = torch.from_numpy(synth.source_row(n, n, h, 3)).cuda()
    cyc = {}
    for precision in ("fp64", "mixed"):
        s = hm.Solver(n, n, h, kk, 1 / k, smoother="gmres3", nu_pre=nu, nu_post=nu, precision=precision, batch=3, **kw)
        x, st, cyc[precision], rr = s.solve(b, tol=tol)
        assert st == hm.MG_OK
        s.close()
    for a, c in zip(cyc["mixed"], cyc["fp64"]):
        assert abs(a - c) <= max(2, 0.1 * c), cyc
