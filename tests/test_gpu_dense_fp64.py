"""The FP64 dense products (8 x 8 gram tiles over split points, the outer
product with its triangular form) at the edges of their tiles: orbital and band
counts around multiples of 8 and 16, real and complex, point counts that are
not multiples of the 32-point stage times the splits, padded vectors.

Tolerance: FP64 sums of at most 20^3 terms, 1e-10 relative as in the other FP64
parity tests.
"""
import math

import numpy as np
import pytest

import oracle
from paper_1601_07159_gb300 import synth
from tests.conftest import rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10

CASES = [("r64", 8, 1, 1, 0), ("r64", 12, 8, 9, 0), ("r64", 12, 17, 5, 4), ("c128", 8, 7, 16, 0), ("c128", 12, 9, 17, 2),
         ("c128", 12, 33, 3, 0), ("c128", 20, 16, 8, 0)]


@pytest.fixture(scope="module")
def ace():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_07159_gb300 import build_lib
    build_lib.build()
    from paper_1601_07159_gb300 import ace as mod
    return mod


@pytest.mark.parametrize("dtype,n,nocc,nb,pad", CASES)
def test_dense_products_match_oracle(ace, dtype, n, nocc, nb, pad):
    L = 0.45 * n
    s = synth.System(n=n, L=L, n_occ=nocc, n_bands=nb, real=dtype == "r64", kernel="erfc", omega=0.3)
    ecut = 0.3 * (math.pi * n / L) ** 2
    phi, psi = synth.orbitals(s, 50 + nocc, ecut=ecut), synth.targets(s, 50 + nocc, ecut=ecut)
    ref = oracle.ace_build(phi, oracle.coulomb_kernel((n,) * 3, (L,) * 3, "erfc", 0.3), s.dv)
    plan = ace.Plan(n, L, nocc, dtype=dtype, kernel="erfc", omega=0.3, ld=s.ng + pad if pad else 0)
    phi_d, psi_d = plan.empty(nocc), plan.empty(nb)
    phi_d.copy_(torch.from_numpy(phi))
    psi_d.copy_(torch.from_numpy(psi))
    out = plan.build(phi_d)
    assert plan.status() == (0, 0)
    host = lambda t: t.cpu().numpy()   # noqa: E731
    assert rel(host(out["M"]), ref["M"]) < TOL
    assert rel(host(out["Xi"]), ref["Xi"]) < TOL
    want = oracle.ace_apply(ref["Xi"], psi, s.dv)
    assert rel(host(plan.apply(out["Xi"], psi_d)), want) < TOL
    y = plan.empty(nb)
    assert rel(host(plan.apply_static(out["Xi"], psi_d, y)), want) < TOL
