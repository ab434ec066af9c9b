"""The FP16-pair apply of complex FP32 plans (grids of 2^16 points or calls of 7 2^18 values and more) at the
edges of its tiles: orbital counts around the 16 of a K chunk and the 128 of a
row tile, band counts that take each MMA width (64, 128, 192 and 256 columns) and
leave a partial last tile, a point count that is not a multiple of 128,
padded vectors, vectors of very different scales, one call below the line, one whose
splits the workspace bounds; against
the oracle and the TF32-split apply.

Tolerance: operands keep 22 bits (2^-23 rounding) of every value down to 2^-18 of
its vector's largest, the dropped product is below 2^-24, and the FP32 sums
truncate at 2^-23 per group of 24 terms in random directions: 1e-5 per band, as in
the other FP32 apply tests, and twice that between two such results.
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5

CASES = [((48, 48, 48), 16, 24, 0), ((48, 48, 48), 1, 1, 0), ((48, 48, 48), 17, 33, 0), ((48, 48, 48), 130, 3, 2), ((36, 36, 36), 1, 97, 0),
         ((36, 36, 36), 33, 96, 6), ((20, 20, 36), 100, 200, 0), ((48, 40, 36), 128, 129, 0), ((32, 32, 32), 15, 200, 0),
         ((24, 24, 24), 20, 30, 0),
         ((36, 36, 36), 300, 300, 0)]


@pytest.fixture(scope="module")
def ace():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_07159_gb300 import build_lib
    build_lib.build()
    from paper_1601_07159_gb300 import ace as mod
    return mod


@pytest.mark.parametrize("grid,nocc,nb,pad", CASES)
def test_apply_matches_oracle_and_tf32(ace, grid, nocc, nb, pad):
    rng = np.random.default_rng(1000 * nocc + nb)
    ng = grid[0] * grid[1] * grid[2]

    def vectors(n, lo, hi):
        v = rng.standard_normal((n, *grid[::-1], 2), dtype=np.float32).view(np.complex64)[..., 0]
        return (v * np.logspace(lo, hi, n)[:, None, None, None]).astype(np.complex64)

    xi, psi = vectors(nocc, -6, 3), vectors(nb, 4, -9)
    out = {}
    for prec in ("default", "split_tf32"):
        plan = ace.Plan(grid, tuple(0.43 * g for g in grid), nocc, dtype="c64", prec=prec, ld=ng + pad if pad else 0)
        xi_d, psi_d, y = plan.empty(nocc), plan.empty(nb), plan.empty(nb)
        xi_d.copy_(torch.from_numpy(xi))
        psi_d.copy_(torch.from_numpy(psi))
        plan.apply(xi_d, psi_d, out=y)
        assert plan.status() == (0, 0)
        out[prec] = y.cpu().numpy().astype(np.complex128)
    want = oracle.ace_apply(xi.astype(np.complex128), psi.astype(np.complex128), plan.dv)
    norm = np.linalg.norm(want.reshape(nb, -1), axis=1)
    err = lambda a, b: float((np.linalg.norm((a - b).reshape(nb, -1), axis=1) / norm).max())   # noqa: E731
    assert err(out["default"], want) < TOL
    assert err(out["default"], out["split_tf32"]) < 2 * TOL
