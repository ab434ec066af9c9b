"""The apply of complex FP32 plans on vectors at the limits of what its FP16 operand
pairs and tensor maps take, on a grid that runs them (2^16 points or more): against
the oracle.
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GRID = (40, 48, 36)
DV = 0.43 ** 3
TOL = 1e-5    # per band, as in the other FP32 apply tests


@pytest.fixture(scope="module")
def ace():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_07159_gb300 import build_lib
    build_lib.build()
    from paper_1601_07159_gb300 import ace as mod
    return mod


def _plan(ace, nocc, **kw):
    return ace.Plan(GRID, tuple(0.43 * g for g in GRID), nocc, dtype="c64", **kw)


def _random(rng, n):
    return rng.standard_normal((n, *GRID[::-1], 2), dtype=np.float32).view(np.complex64)[..., 0]


def _apply(plan, xi, psi):
    y = plan.apply(torch.from_numpy(xi).cuda(), torch.from_numpy(psi).cuda(), out=torch.empty(psi.shape, dtype=torch.complex64, device="cuda"))
    assert plan.status() == (0, 0)
    return y.cpu().numpy().astype(np.complex128)


def _want(xi, psi):
    return oracle.ace_apply(xi.astype(np.complex128), psi.astype(np.complex128), DV)


@pytest.mark.parametrize("ld", [1 << 36, 1 << 37, 1 << 40])
def test_strides_beyond_a_tensor_map(ace, ld):
    """One orbital, one band: the distance to a next vector is never used, so any is
    taken. A tensor map's is below 2^40 bytes (2^37 elements)."""
    rng = np.random.default_rng(1)
    xi, psi = _random(rng, 1), _random(rng, 1)
    got, want = _apply(_plan(ace, 1, ld=ld), xi, psi), _want(xi, psi)
    assert np.linalg.norm(got - want) < TOL * np.linalg.norm(want)


def _near(rng, n, decades, axis_up=False):
    """n vectors that share an envelope falling by `decades` along the last grid axis (rising
    with axis_up), within a factor of two of it at every point: overlaps without
    cancellation, so that an error per point shows."""
    z = np.arange(GRID[2]) / (GRID[2] - 1)
    env = 10.0 ** (-decades * (1 - z if axis_up else z))[None, :, None, None]
    noise = rng.uniform(-0.5, 0.5, (n, *GRID[::-1])) + 1j * rng.uniform(-0.5, 0.5, (n, *GRID[::-1]))
    return (env * (1.0 + noise)).astype(np.complex64)


def _point_error(got, xi, psi):
    """The largest error of a value over sum_k |Xi_k(r)| |C_kb|, its terms' size."""
    x, p = xi.astype(np.complex128).reshape(len(xi), -1), psi.astype(np.complex128).reshape(len(psi), -1)
    c = DV * (x.conj() @ p.T)
    size = np.abs(c).T @ np.abs(x)
    return float((np.abs(got.reshape(size.shape) + c.T @ x) / size).max())


# The same bounds per value as per band: operands keep 22 bits of a value beside its
# neighbours, the FP32 sums truncate at 2^-23 per group of 24 terms; 1e-5 as above.
@pytest.mark.parametrize("nocc,nb", [(5, 3), (17, 40), (140, 100)])
@pytest.mark.parametrize("prec", ["default", "split_tf32"])
def test_accuracy_where_every_orbital_is_small(ace, prec, nocc, nb):
    """Vacuum: every orbital decays by ten decades. The values there come as accurate,
    relative to the orbitals there, as elsewhere."""
    rng = np.random.default_rng(nocc)
    xi, psi = _near(rng, nocc, 10.0), _near(rng, nb, 10.0)
    assert _point_error(_apply(_plan(ace, nocc, prec=prec), xi, psi), xi, psi) < TOL


@pytest.mark.parametrize("decades", [5.0, 10.0])
@pytest.mark.parametrize("nocc,nb", [(5, 3), (17, 40), (140, 100)])
@pytest.mark.parametrize("prec", ["default", "split_tf32"])
def test_accuracy_of_overlaps_in_the_tails(ace, prec, nocc, nb, decades):
    """Bands that grow where the orbitals decay: every point contributes alike to C, from
    values far below the largest of both vectors."""
    rng = np.random.default_rng(nocc + 1)
    xi, psi = _near(rng, nocc, decades), _near(rng, nb, decades, axis_up=True)
    got, want = _apply(_plan(ace, nocc, prec=prec), xi, psi), _want(xi, psi)
    err = np.linalg.norm((got - want).reshape(nb, -1), axis=1) / np.linalg.norm(want.reshape(nb, -1), axis=1)
    print(prec, nocc, nb, decades, err.max())
    assert err.max() < TOL


def test_vectors_of_subnormal_size(ace):
    """Orbitals below FP32's normal range on bands near its top: every intermediate
    leaves the range, the result does not (and carries the subnormals' spacing, 2^-149)."""
    rng = np.random.default_rng(5)
    xi, psi = _random(rng, 6) * np.float32(1e-39), _random(rng, 5) * np.float32(5e37)
    got, want = _apply(_plan(ace, 6), xi, psi), _want(xi, psi)
    err = np.linalg.norm((got - want).reshape(5, -1), axis=1)
    assert (err < TOL * np.linalg.norm(want.reshape(5, -1), axis=1) + 2.0 ** -149 * np.sqrt(2 * got[0].size)).all()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_values_stay_in_their_band(ace, bad):
    """A band with a NaN or an infinity has no finite result; the others are those
    without it. In an orbital it reaches every band."""
    rng = np.random.default_rng(6)
    xi, psi = _random(rng, 20), _random(rng, 30)
    clean = _apply(_plan(ace, 20), xi, psi)
    psi[7, 3, 5, 9] = bad
    got = _apply(_plan(ace, 20), xi, psi)
    assert not np.isfinite(got[7]).any()
    assert np.array_equal(np.delete(got, 7, 0), np.delete(clean, 7, 0))
    psi[7, 3, 5, 9] = 0
    xi[4, 1, 2, 3] = bad
    assert not np.isfinite(_apply(_plan(ace, 20), xi, psi)).any()
