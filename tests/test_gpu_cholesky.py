"""The blocked FP64 Cholesky factorisation and inverse of -M at the edges of its
16-column panels, 8 x 8 tiles and doubling levels (levels with a lone, a full and
a ragged last block): Xi and M of FP64 builds against the oracle.

Tolerance: random orbitals give a well-conditioned -M (condition below 1e4), so
the factor's rounding error stays far below 1e-10 relative, the tolerance of the
other FP64 parity tests.
"""
import numpy as np
import pytest

import oracle
from tests.conftest import rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.fixture(scope="module")
def ace():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_07159_gb300 import build_lib
    build_lib.build()
    from paper_1601_07159_gb300 import ace as mod
    return mod


@pytest.mark.parametrize("nocc", [2, 15, 16, 17, 31, 32, 33, 49, 63, 64, 65, 80, 97, 129])
def test_factor_and_inverse_match_oracle(ace, nocc):
    n, L = 12, 5.4
    rng = np.random.default_rng(nocc)
    phi = rng.standard_normal((nocc, n, n, n)) + 1j * rng.standard_normal((nocc, n, n, n))
    phi /= np.sqrt(n ** 3)
    ref = oracle.ace_build(phi, oracle.coulomb_kernel((n,) * 3, (L,) * 3, "erfc", 0.3), (L / n) ** 3)
    plan = ace.Plan(n, L, nocc, dtype="c128", kernel="erfc", omega=0.3)
    phi_d = plan.empty(nocc)
    phi_d.copy_(torch.from_numpy(phi))
    out = plan.build(phi_d)
    assert plan.status() == (0, 0)
    assert rel(out["M"].cpu().numpy(), ref["M"]) < TOL
    assert rel(out["Xi"].cpu().numpy(), ref["Xi"]) < TOL
