"""The pivot that a failed factorisation reports: a zero orbital makes its row and
column of M, and so its pivot, exactly zero. Positions through a 16-column panel, at
panel edges and in a ragged last panel; many times each, as the verdict is passed
between warps.
"""
import pytest

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
