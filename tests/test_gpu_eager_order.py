"""Eager calls (graphs off) right behind the kernel that writes their vectors: pass A
reads them before its programmatic wait, so the call's first pass A must depend on
that kernel in full, while the passes of the call stay chained.

The results have to be those of the same calls with a synchronisation in between, to
the bit: the same kernels on the same values.
"""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# grid, dtype: whole-line planes and (c64 from 96, FP64 from 64) two-lane planes
CASES = [((16, 16, 16), "c64"), ((48, 48, 48), "c64"), ((96, 96, 8), "c64"), ((24, 24, 24), "c128"), ((64, 64, 8), "c128"),
         ((20, 20, 20), "r64"), ((64, 64, 12), "r64")]


@pytest.fixture(scope="module")
def ace():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_07159_gb300 import build_lib
    build_lib.build()
    from paper_1601_07159_gb300 import ace as mod
    return mod


def _plan(ace, grid, dtype):
    return ace.Plan(grid, tuple(0.45 * n for n in grid), 4, dtype=dtype, kernel="bare", graphs=False)


def _field(plan, count, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rt = torch.float32 if plan.dtype == "c64" else torch.float64
    x = torch.randn((count, *plan.shape, 1 if plan.dtype == "r64" else 2), generator=gen, device="cuda", dtype=rt)
    return x[..., 0].contiguous() if plan.dtype == "r64" else torch.view_as_complex(x)


@pytest.mark.parametrize("grid,dtype", CASES)
def test_back_to_back_equals_synchronised(ace, grid, dtype):
    plan = _plan(ace, grid, dtype)
    base = _field(plan, 3, 5)

    def chain(i, wait):
        sync = torch.cuda.synchronize if wait else lambda: None
        rho = base * (1.0 + 0.125 * i)          # a fresh tensor, written by the kernel in front of the call
        sync()
        v = plan.poisson(rho)
        sync()
        u = plan.poisson(v)                     # behind the pass C that writes its density
        sync()
        y = plan.exchange_apply(_orbitals, u)
        sync()
        e, _ = plan.energy_grad(_orbitals * (1.0 + 0.125 * i))
        sync()
        return v, u, y, e

    _orbitals = _field(plan, 4, 9)
    for i in range(20):
        got, want = chain(i, False), chain(i, True)
        for a, b in zip(got, want):
            assert torch.equal(a, b)


class _EdgeData(ctypes.Structure):
    _fields_ = [("from_port", ctypes.c_ubyte), ("to_port", ctypes.c_ubyte), ("type", ctypes.c_ubyte),
                ("reserved", ctypes.c_ubyte * 5)]


@pytest.mark.parametrize("grid,dtype", CASES[:2] + CASES[4:5])
def test_first_pass_depends_in_full(ace, grid, dtype):
    """The captured form of [kernel that writes rho, eager Poisson call]: the edge from
    that kernel is a full one, the edges between the passes are programmatic."""
    rt = ctypes.CDLL("libcudart.so.13")
    plan = _plan(ace, grid, dtype)
    src = _field(plan, 2, 3)
    rho, v = torch.empty_like(src), torch.empty_like(src)
    stream = torch.cuda.Stream()
    graph = ctypes.c_void_p()
    with torch.cuda.stream(stream):
        torch.add(src, src, out=rho)
        stream.synchronize()
        plan.poisson(rho, out=v)                # schedule and workspace of this call
        stream.synchronize()
        handle = ctypes.c_void_p(stream.cuda_stream)
        assert rt.cudaStreamBeginCapture(handle, 2) == 0      # relaxed
        torch.add(src, src, out=rho)
        plan.poisson(rho, out=v)
        assert rt.cudaStreamEndCapture(handle, ctypes.byref(graph)) == 0
    n = ctypes.c_size_t(0)
    assert rt.cudaGraphGetEdges(graph, None, None, None, ctypes.byref(n)) == 0
    src_nodes, dst_nodes, data = (ctypes.c_void_p * n.value)(), (ctypes.c_void_p * n.value)(), (_EdgeData * n.value)()
    assert rt.cudaGraphGetEdges(graph, src_nodes, dst_nodes, data, ctypes.byref(n)) == 0
    rt.cudaGraphDestroy(graph)
    edges = {src_nodes[i]: (dst_nodes[i], data[i].type) for i in range(n.value)}
    assert len(edges) == n.value == 3           # add -> A -> B -> C
    node = (set(edges) - {d for d, _ in edges.values()}).pop()
    types = []
    while node in edges:
        node, t = edges[node]
        types.append(t)
    assert types == [0, 1, 1]
