"""FP64 plans: a workspace sized for a block of vectors serves every narrower block
(the sizes never fall as the block grows), as a program that allocates once for its
widest block relies on.
"""
import ctypes

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


@pytest.mark.parametrize("n,nocc", [(8, 1), (12, 8), (24, 17), (48, 33)])
@pytest.mark.parametrize("dtype", ["r64", "c128"])
def test_sizes_do_not_fall(ace, dtype, n, nocc):
    plan = ace.Plan(n, 0.45 * n, nocc, dtype=dtype)
    for op, lo in ((ace.OP_APPLY, 1), (ace.OP_BUILD_OVERSAMPLED, nocc)):
        sizes = [plan.workspace_size(op, nb) for nb in range(lo, lo + 140)]
        assert sizes == sorted(sizes)


def test_narrower_block_in_a_wider_workspace(ace):
    plan = ace.Plan(24, 10.0, 8, dtype="c128")
    gen = torch.Generator(device="cuda").manual_seed(2)
    xi = torch.randn((8, *plan.shape), generator=gen, device="cuda", dtype=torch.complex128)
    psi = torch.randn((32, *plan.shape), generator=gen, device="cuda", dtype=torch.complex128)
    ws = torch.empty(plan.workspace_size(ace.OP_APPLY, 33), dtype=torch.uint8, device="cuda")
    y = torch.empty_like(psi)
    p = lambda t: ctypes.c_void_p(t.data_ptr())   # noqa: E731
    assert ace.lib().ace_apply(plan._h, p(xi), p(psi), 32, p(y), p(ws), ws.numel(), None) == ace.ACE_OK
    assert torch.equal(y, plan.apply(xi, psi))


@pytest.mark.parametrize("lanes", [2, 3])
def test_one_chain_takes_one_buffer(ace, lanes):
    """C64 plans run their passes as one chain in one scratch buffer; a tuned schedule's
    lanes (which belong to the form without overlap) add none."""
    for op in (ace.OP_BUILD, ace.OP_ENERGY_GRAD, ace.OP_EXCHANGE_APPLY):
        plans = [ace.Plan(24, 10.0, 20, dtype="c64", max_pairs=64, lanes=k) for k in (0, lanes)]
        assert plans[0].workspace_size(op, 5) == plans[1].workspace_size(op, 5)
    spread = ace.Plan(24, 10.0, 20, dtype="c64", max_pairs=64, lanes=lanes, overlap=False)
    assert spread.workspace_size(ace.OP_BUILD) > plans[0].workspace_size(ace.OP_BUILD)
    assert spread.effective_schedule()["lanes"] == lanes
