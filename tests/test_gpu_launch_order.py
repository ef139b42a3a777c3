"""What the first launch of an evolution may start before.

A sweep reads its tables before it waits for the launch before it (programmatic dependent
launch), so only a sweep behind another one may be launched that way: the first launch of an
evolution or of a batch can follow the kernel that writes those tables.  The launches are
captured behind a kernel of the caller and the graph's edges looked at; nothing runs.
"""
import ctypes

import numpy as np
import pytest

from paper_2606_16959_gb300 import hs, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_16959_gb300 import _build
    _build.build()
    hs.lib()


class _Edge(ctypes.Structure):
    _fields_ = [("from_port", ctypes.c_ubyte), ("to_port", ctypes.c_ubyte), ("type", ctypes.c_ubyte),
                ("reserved", ctypes.c_ubyte * 5)]


PROGRAMMATIC = 1  # CU_GRAPH_DEPENDENCY_TYPE_PROGRAMMATIC


def _edge_types(graph):
    """The edges' types in the order of a captured chain of nodes."""
    cu = ctypes.CDLL("libcuda.so.1")
    n = ctypes.c_size_t(0)
    g = ctypes.c_void_p(graph)
    assert cu.cuGraphGetEdges_v2(g, None, None, None, ctypes.byref(n)) == 0
    src, dst, data = (ctypes.c_void_p * n.value)(), (ctypes.c_void_p * n.value)(), (_Edge * n.value)()
    assert cu.cuGraphGetEdges_v2(g, src, dst, data, ctypes.byref(n)) == 0
    nxt = {a: (b, d.type) for a, b, d in zip(src, dst, data)}
    assert len(nxt) == n.value  # a chain
    at = (set(src) - set(dst)).pop()
    types = []
    while at in nxt:
        at, t = nxt[at]
        types.append(t)
    return types


def _captured(call, psi):
    call()  # first use of every kernel, outside the capture
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        psi.mul_(1.0)  # stands for whatever wrote the tables
        call()
    return _edge_types(g.raw_cuda_graph())


@pytest.mark.parametrize("kind,method,dt", [("tfim", "FUSED", "c64"), ("tfim", "REG", "c64"), ("tfim", "REG", "c128"),
                                            ("heisenberg", "FUSED", "c128"), ("heisenberg", "AUTO", "c64")])
def test_first_sweep_waits(kind, method, dt):
    n = 15  # (more than a tile: several sweeps)
    ham = W.tfim_chain(n, 1.0, 0.7) if kind == "tfim" else W.heisenberg_chain(n, np.full(n, 0.8))
    f = hs.hs_build_factors(ham.labels, ham.coeffs, 1.0, 4, 4, dt)
    psi = torch.zeros(1 << n, dtype=torch.complex64 if dt == "c64" else torch.complex128, device="cuda")
    types = _captured(lambda: hs.hs_evolve_ex(f, psi, 8, method=getattr(hs, "HS_METHOD_" + method)), psi)
    assert len(types) >= 2
    assert types[0] != PROGRAMMATIC
    assert all(t == PROGRAMMATIC for t in types[1:])


@pytest.mark.parametrize("method", [0, hs.HS_METHOD_REG])
def test_first_batch_level_waits(method):
    jobs = []
    for n in (14, 15):
        ham = W.tfim_chain(n, 1.0, 0.7)
        f = hs.hs_build_factors(ham.labels, ham.coeffs, 1.0, 4, 4, "c64")
        jobs.append((f, torch.zeros(1 << n, dtype=torch.complex64, device="cuda"), 4))
    b = hs.hs_batch_create(jobs, method=method, use_graph=False)
    types = _captured(lambda: hs.hs_batch_launch(b), jobs[0][1])
    first = 2 if method == hs.HS_METHOD_REG else 1  # (a register batch writes its tables first)
    assert len(types) > first
    assert all(t != PROGRAMMATIC for t in types[:first])
    assert all(t == PROGRAMMATIC for t in types[first:])
