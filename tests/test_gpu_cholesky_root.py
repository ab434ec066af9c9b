"""The diagonal of the Cholesky factor is CUDA's correctly rounded square root and
division: with one orbital, Xi = W (1 / sqrt(-M)), so the returned M and W give Xi to
the bit, over the exponent range of M.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ace():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_07159_gb300 import build_lib
    build_lib.build()
    from paper_1601_07159_gb300 import ace as mod
    return mod


def test_root_and_reciprocal_are_correctly_rounded(ace):
    rng = np.random.default_rng(11)
    plan = ace.Plan(8, 3.6, 1, dtype="r64", kernel="erfc", omega=0.3)
    phi_d = plan.empty(1)
    for e in np.linspace(-70.0, 70.0, 60):           # M is of the fourth power
        phi_d.copy_(torch.from_numpy(rng.standard_normal((1, 8, 8, 8)) * 10.0 ** e))
        out = plan.build(phi_d)
        assert plan.status() == (0, 0)
        m, w = out["M"].cpu().numpy()[0, 0], out["W"].cpu().numpy()
        assert np.array_equal(out["Xi"].cpu().numpy(), w * (1.0 / np.sqrt(-m)))
