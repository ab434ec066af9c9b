"""Every way of running the pair passes of many small batches gives the bits of eager
launches, in each dtype: the one-stream chain of C64 plans, the two-stream form of FP64
plans (pass A of a batch beside pass D of the one before, two scratch buffers in turn),
and a round's batches spread over lanes. Builds, V_X on other vectors, and the
Poisson solves (passes A, B and C alone) with several batches; capture and replay.
"""
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


@pytest.mark.parametrize("kw", [{}, {"lanes": 3, "overlap": False}, {"pdl": False}])
@pytest.mark.parametrize("dtype", ["c64", "c128", "r64"])
def test_schedules_match_eager(ace, dtype, kw):
    n, nocc, nb = 24, 21, 23
    opts = dict(dtype=dtype, kernel="erfc", omega=0.3, tile=4, max_pairs=16)
    eager = ace.Plan(n, 10.0, nocc, graphs=False, **opts)
    other = ace.Plan(n, 10.0, nocc, **opts, **kw)
    gen = torch.Generator(device="cuda").manual_seed(4)
    phi, psi = (torch.randn((k, *eager.shape), generator=gen, device="cuda", dtype=eager.tdtype) for k in (nocc, nb))
    want = eager.build(phi)
    want_y, want_v, want_e = eager.exchange_apply(phi, psi), eager.poisson(psi), eager.energy_grad(phi, grad=True)
    assert eager.status() == (0, 0)
    xi, w, y, v, g = other.empty(nocc), other.empty(nocc), other.empty(nb), other.empty(nb), other.empty(nocc)
    for _ in range(3):                          # capture, then replay
        for t in (xi, w, y, v, g):
            t.fill_(float("nan"))
        got = other.build(phi, xi=xi, w=w)
        assert torch.equal(got["W"], want["W"]) and torch.equal(got["M"], want["M"]) and torch.equal(xi, want["Xi"])
        assert torch.equal(other.exchange_apply(phi, psi, out=y), want_y)
        assert torch.equal(other.poisson(psi, out=v), want_v)
        e, _ = other.energy_grad(phi, grad=True, out=g)
        assert torch.equal(g, want_e[1])
        # the energy's partial sums are kept per lane: their order differs
        assert abs(e.item() - want_e[0].item()) <= 1e-13 * abs(want_e[0].item())
        assert other.status() == (0, 0)
