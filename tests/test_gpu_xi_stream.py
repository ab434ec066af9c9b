"""The slice product of Xi as one stream of chunks per block: orbital counts that
give tiles of one to several chunks and accumulator groups (16 orbitals a chunk, 64
a group, 48 columns a tile), on a grid with fewer tiles than blocks and one with
several tiles per block.

The product is exact up to its documented truncation (five 8-bit digits per
operand, digit pairs of weight six or less) and one final rounding, so it is
compared bit for bit with the same sums in host integer arithmetic, in FP64 and
FP32 output. L^{-*} is read off the plain FP64 product of unit vectors.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BETA, T = 8, 6


@pytest.fixture(scope="module")
def ace():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_07159_gb300 import build_lib
    build_lib.build()
    from paper_1601_07159_gb300 import ace as mod
    return mod


def _digits(x, e):
    """The T - 1 signed digits of x 2^-e."""
    x, out = np.ldexp(x, BETA - e), []
    for _ in range(T - 1):
        out.append(np.rint(x))
        x = (x - out[-1]) * 2 ** BETA
    return out


def _exponent(m):
    return np.where(m > 0, np.frexp(m)[1], 0)


def _slice_sums(w, c):
    """w [nk][ng], c [nk][nb] complex: integer sums of Re and Im Xi [ng][nb] and their exponents."""
    nk, nb = c.shape
    a = np.empty((w.shape[1], 2 * nk))
    a[:, 0::2], a[:, 1::2] = w.real.T, w.imag.T
    b = np.empty((2 * nk, 2 * nb))
    b[0::2, :nb], b[1::2, :nb], b[0::2, nb:], b[1::2, nb:] = c.real, -c.imag, c.imag, c.real
    e, f = _exponent(np.abs(a).max(1)), _exponent(np.abs(b).max(0))
    da, db = _digits(a, e[:, None]), _digits(b, f[None, :])
    s = np.zeros((a.shape[0], 2 * nb), dtype=np.int64)
    for wt in range(2, T + 1):
        p = sum(da[i - 1] @ db[wt - i - 1] for i in range(1, wt))
        s += p.astype(np.int64) << (BETA * (T - wt))
    return s, e[:, None] + f[None, :] - BETA * T


@pytest.mark.parametrize("n", [8, 36])
@pytest.mark.parametrize("nocc", [1, 16, 17, 48, 49, 65, 97])
def test_slices_match_integer_sums(ace, n, nocc):
    rng = np.random.default_rng(nocc)
    phi = rng.standard_normal((nocc, n, n, n, 2), dtype=np.float32).view(np.complex64)[..., 0] / np.float32(n ** 1.5)
    plan = ace.Plan(n, 0.45 * n, nocc, dtype="c64", kernel="erfc", omega=0.3)
    phi_d, unit = plan.empty(nocc), plan.empty(nocc)
    phi_d.copy_(torch.from_numpy(phi))
    out = plan.build(phi_d)
    assert plan.status() == (0, 0)
    unit.zero_()
    for k in range(nocc):
        unit[k].view(-1)[k] = 1
    c = plan.debug_xi_product(unit, 2).reshape(nocc, -1)[:, :nocc].T.cpu().numpy()
    s, e = _slice_sums(out["W"].reshape(nocc, -1).cpu().numpy().astype(np.complex128), c)
    want = np.ldexp(s.astype(np.float64), e)
    want32 = np.ldexp(s.astype(np.float32), e)
    for got, ref in ((plan.debug_xi_product(out["W"], 1), want), (out["Xi"], want32)):
        got = got.reshape(nocc, -1).T.cpu().numpy()
        assert np.array_equal(got.real, ref[:, :nocc]) and np.array_equal(got.imag, ref[:, nocc:])
