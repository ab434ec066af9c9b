"""The pivot that a failed factorisation reports: a zero orbital makes its row and
column of M, and so its pivot, exactly zero. Positions through a 16-column panel, at
panel edges and in a ragged last panel; many times each, as the verdict is passed
between warps. And pivots of matrices far from order one.
"""
import numpy as np
import pytest

import oracle
from tests.conftest import rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 40


@pytest.fixture(scope="module")
def ace():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_07159_gb300 import build_lib
    build_lib.build()
    from paper_1601_07159_gb300 import ace as mod
    return mod


@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_reported_pivot(ace, dtype):
    plan = ace.Plan(8, 3.6, N, dtype=dtype, kernel="erfc", omega=0.3)
    gen = torch.Generator(device="cuda").manual_seed(7)
    good = torch.randn((N, *plan.shape), generator=gen, device="cuda", dtype=plan.tdtype) / 16
    xi = plan.empty(N)
    plan.build(good, xi=xi)
    assert plan.status() == (0, 0)
    phi = plan.empty(N)
    for p in (0, 1, 2, 3, 8, 13, 14, 15, 16, 17, 30, 31, 32, 38, 39):
        phi.copy_(good)
        phi[p] = 0
        for _ in range(40):
            plan.build(phi, want_w=False, want_m=False, xi=xi)
            assert plan.status() == (ace.ACE_ERR_NOT_POSDEF, p + 1)
    plan.build(good, xi=xi)
    assert plan.status() == (0, 0)


@pytest.mark.parametrize("dtype", ["c128", "r64"])
@pytest.mark.parametrize("scale", [1e-45, 1e-30, 1e30, 1e45])
def test_pivots_over_the_exponent_range(ace, dtype, scale):
    """M is of the fourth power of the orbitals: entries near 1e-180 and 1e180 are
    ordinary numbers, their squares are not. Xi is of the first power, and must agree
    with that of the unscaled orbitals to the tolerance of the FP64 parity tests."""
    n, nocc, L = 8, 20, 3.6
    rng = np.random.default_rng(3)
    phi = rng.standard_normal((nocc, n, n, n)) + (1j * rng.standard_normal((nocc, n, n, n)) if dtype == "c128" else 0)
    ref = oracle.ace_build(phi, oracle.coulomb_kernel((n,) * 3, (L,) * 3, "erfc", 0.3), (L / n) ** 3)
    plan = ace.Plan(n, L, nocc, dtype=dtype, kernel="erfc", omega=0.3)
    phi_d = plan.empty(nocc)
    phi_d.copy_(torch.from_numpy(phi * scale))
    out = plan.build(phi_d)
    assert plan.status() == (0, 0)
    assert rel(out["Xi"].cpu().numpy() / scale, ref["Xi"]) < 1e-10
