"""mg_profile(what = 4) for every value of the march option: the bytes are those
of the Arnoldi form of the step for the kernels that the cycle runs, as the
header says: on the fine level row marches in complex64 unless march = 0 (13
vector passes, else 23), in complex128 only with march = 1 (16, else 28); on a
Kronecker-form level column marches unless march = 0 (complex64 19, else 23;
complex128 28 either way)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2308_13476_gb300 as hm  # noqa: E402


@pytest.mark.parametrize("precision,march,fine,level1", [
    ("mixed", -1, 13, 19), ("mixed", 1, 13, 19), ("mixed", 0, 23, 23), ("mixed-ff", -1, 13, 19),
    ("fp64", -1, 28, 28), ("fp64", 1, 16, 28), ("fp64", 0, 28, 28)])
def test_gmres_step_bytes(precision, march, fine, level1):
    n, B = 64, 2
    s = hm.Solver(n, n, 1.0 / n, 20.0, 0.05, smoother="gmres3", nu_pre=2, nu_post=2, precision=precision, batch=B,
                  march=march)
    e = 16 if precision == "fp64" else 8
    for level, passes in ((0, fine), (1, level1)):
        ms, nbytes = s.profile(4, level, reps=2)
        assert ms > 0 and nbytes == pytest.approx(passes * e * B * (n // 2**level + 1) ** 2, rel=1e-9), level
    s.close()
