"""Pass D of FP32 plans on full off-diagonal tiles (four threads per grid point,
the right outputs' sums handed from one half of the left orbitals to the other)
against the FP64 oracle: W and the stored-potential gradient at the smallest
and odd point counts, with full tiles alone, beside ragged ones, and with
padded vectors.

Tolerance: W_i is a sum of N FP32 products v phi; each carries a few FP32
roundings of the transforms (about 2^-22 of its size), so 1e-6 relative bounds
it with room, as in the other FP32 parity tests.
"""
import math

import numpy as np
import pytest

import oracle
from paper_1601_07159_gb300 import synth
from tests.conftest import rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-6

# grid, N, extra elements between vectors: 512 points (a tile's last block is its only one), 1728, 2880
# (orthorhombic), 8000; N = 16: one full off-diagonal tile; 17, 27: beside ragged ones; 40: five blocks
CASES = [((8, 8, 8), 16, 0), ((8, 8, 8), 17, 2), ((12, 12, 12), 27, 0), ((12, 12, 20), 16, 6), ((20, 20, 20), 24, 0),
         ((12, 16, 8), 40, 0)]


@pytest.fixture(scope="module")
def ace():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_07159_gb300 import build_lib
    build_lib.build()
    from paper_1601_07159_gb300 import ace as mod
    return mod


@pytest.mark.parametrize("grid,nocc,pad", CASES)
def test_full_tiles_match_oracle(ace, grid, nocc, pad):
    cell = tuple(0.45 * n for n in grid)
    s = synth.System(n=0, L=0.0, n_occ=nocc, n_bands=1, kernel="erfc", omega=0.3, grid=grid, cell=cell)
    ecut = 0.3 * min((math.pi * n / l) ** 2 for n, l in zip(grid, cell))
    rng = np.random.Generator(np.random.PCG64(77 + nocc))
    phi = synth.targets(s, 77 + nocc, count=nocc, ecut=ecut) * rng.uniform(0.5, 2.0, nocc)[:, None, None, None]
    kern = oracle.coulomb_kernel(s.shape, s.lengths, "erfc", 0.3)
    ref = oracle.exchange_W(phi, kern)

    plan = ace.Plan(grid, cell, nocc, dtype="c64", kernel="erfc", omega=0.3, ld=s.ng + pad if pad else 0)
    phi_d, w = plan.empty(nocc), plan.empty(nocc)
    phi_d.copy_(torch.from_numpy(phi).to(torch.complex64))
    phi64 = phi_d.cpu().numpy().astype(np.complex128)
    assert rel(phi64, phi) < 1e-7
    plan.build(phi_d, w=w)
    assert rel(w.cpu().numpy().astype(np.complex128), ref) < TOL

    ex, _ = plan.energy_grad(phi_d, grad=False, recompute=False)
    _, g = plan.energy_grad(phi_d, grad=True, recompute=False)
    assert rel(g.cpu().numpy().astype(np.complex128), 2.0 * s.dv * ref) < TOL
    e_ref = 0.5 * s.dv * float(np.sum((phi.conj() * ref).real))
    assert abs(ex.item() - e_ref) < TOL * abs(e_ref)


# N, n_b, dtype, max_pairs: one-sided tiles with 1-8 right orbitals (one or both halves of pass D, full and
# ragged) and left chunks of every remainder modulo the four orbitals taken at a time
RECT = [(5, 1, "c64", 0), (13, 9, "c64", 64), (7, 4, "c64", 0), (18, 12, "c64", 0), (6, 11, "c128", 64),
        (3, 8, "c64", 0), (9, 5, "c128", 0)]


@pytest.mark.parametrize("nocc,nb,dtype,max_pairs", RECT)
def test_one_sided_tiles_match_oracle(ace, nocc, nb, dtype, max_pairs):
    n, L = 12, 5.4
    s = synth.System(n=n, L=L, n_occ=nocc, n_bands=nb, kernel="erfc", omega=0.3)
    ecut = 0.3 * (math.pi * n / L) ** 2
    phi, psi = synth.orbitals(s, 31 + nocc, ecut=ecut), synth.targets(s, 31 + nocc, ecut=ecut)
    ref = oracle.exchange_apply(phi, psi, oracle.coulomb_kernel((n,) * 3, (L,) * 3, "erfc", 0.3))
    plan = ace.Plan(n, L, nocc, dtype=dtype, kernel="erfc", omega=0.3, max_pairs=max_pairs)
    td = ace.TORCH_DTYPES[dtype]
    y = plan.exchange_apply(torch.from_numpy(phi).to(td).cuda(), torch.from_numpy(psi).to(td).cuda())
    assert rel(y.cpu().numpy().astype(np.complex128), ref) < (TOL if dtype == "c64" else 1e-10)
