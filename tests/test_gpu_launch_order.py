"""What the first launch of an evolution waits for.

A sweep is launched to start while the launch before it runs (programmatic dependent launch),
and reads its tables before it waits for that launch.  The launch before the first one may be
the kernel that writes the tables, so that sweep has to wait before it reads them.  The launches
are captured behind a kernel of the caller, and the graph's edges and the sweeps' first argument
(wait_first) looked at; the graph does not run.
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


class _Kernel(ctypes.Structure):  # CUDA_KERNEL_NODE_PARAMS
    _fields_ = [("func", ctypes.c_void_p), ("dims", ctypes.c_uint * 7), ("params", ctypes.POINTER(ctypes.c_void_p)),
                ("extra", ctypes.c_void_p), ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


PROGRAMMATIC = 1  # CU_GRAPH_DEPENDENCY_TYPE_PROGRAMMATIC


def _chain(graph):
    """A captured chain of kernels: (edge type, first word of the arguments) of all but the first."""
    cu = ctypes.CDLL("libcuda.so.1")
    n = ctypes.c_size_t(0)
    g = ctypes.c_void_p(graph)
    assert cu.cuGraphGetEdges_v2(g, None, None, None, ctypes.byref(n)) == 0
    src, dst, data = (ctypes.c_void_p * n.value)(), (ctypes.c_void_p * n.value)(), (_Edge * n.value)()
    assert cu.cuGraphGetEdges_v2(g, src, dst, data, ctypes.byref(n)) == 0
    nxt = {a: (b, d.type) for a, b, d in zip(src, dst, data)}
    assert len(nxt) == n.value  # a chain
    at = (set(src) - set(dst)).pop()
    out = []
    while at in nxt:
        at, t = nxt[at]
        k = _Kernel()
        assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(at), ctypes.byref(k)) == 0
        out.append((t, ctypes.cast(k.params[0], ctypes.POINTER(ctypes.c_int))[0]))
    return out


def _captured(call, psi):
    call()  # first use of every kernel, outside the capture
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        psi.mul_(1.0)  # stands for whatever wrote the tables
        call()
    return _chain(g.raw_cuda_graph())


@pytest.mark.parametrize("kind,method,dt", [("tfim", "FUSED", "c64"), ("tfim", "REG", "c64"), ("tfim", "REG", "c128"),
                                            ("heisenberg", "FUSED", "c128"), ("heisenberg", "AUTO", "c64")])
def test_first_sweep_waits(kind, method, dt):
    n = 15  # (more than a tile: several sweeps)
    ham = W.tfim_chain(n, 1.0, 0.7) if kind == "tfim" else W.heisenberg_chain(n, np.full(n, 0.8))
    f = hs.hs_build_factors(ham.labels, ham.coeffs, 1.0, 4, 4, dt)
    psi = torch.zeros(1 << n, dtype=torch.complex64 if dt == "c64" else torch.complex128, device="cuda")
    sweeps = _captured(lambda: hs.hs_evolve_ex(f, psi, 8, method=getattr(hs, "HS_METHOD_" + method)), psi)
    assert len(sweeps) >= 2
    assert [w for _, w in sweeps] == [1] + [0] * (len(sweeps) - 1)
    assert all(t == PROGRAMMATIC for t, _ in sweeps)


@pytest.mark.parametrize("method", [0, hs.HS_METHOD_REG])
def test_first_batch_level_waits(method):
    jobs = []
    for n in (14, 15):
        ham = W.tfim_chain(n, 1.0, 0.7)
        f = hs.hs_build_factors(ham.labels, ham.coeffs, 1.0, 4, 4, "c64")
        jobs.append((f, torch.zeros(1 << n, dtype=torch.complex64, device="cuda"), 4))
    b = hs.hs_batch_create(jobs, method=method, use_graph=False)
    types = [t for t, _ in _captured(lambda: hs.hs_batch_launch(b), jobs[0][1])]
    first = 2 if method == hs.HS_METHOD_REG else 1  # (a register batch writes its tables first)
    assert len(types) > first
    assert all(t != PROGRAMMATIC for t in types[:first])
    assert all(t == PROGRAMMATIC for t in types[first:])
