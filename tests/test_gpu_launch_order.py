"""That no sweep reads its tables before the kernel that writes them is complete.

A sweep is launched to start while the launch before it runs (programmatic dependent launch),
and reads its tables before it waits for that launch.  So the launch before the first one must
not be what writes them: a static set's build ends with a memory write that starts behind its
kernels, and the first sweep of a driven set is an ordinary launch.  The launches are captured,
and the graphs' nodes and edges looked at; the graphs do not run.
"""
import os
import subprocess
import sys
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
KERNEL, MEMSET = 0, 2  # CU_GRAPH_NODE_TYPE_*


def chain(graph):
    """A captured chain: (type of the edge to it, node type) of all nodes but the first."""
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
        at, edge = nxt[at]
        kind = ctypes.c_int(-1)
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(at), ctypes.byref(kind)) == 0
        out.append((edge, kind.value))
    return out


def _captured(call, psi):
    call()  # first use of every kernel, outside the capture
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        psi.mul_(1.0)  # stands for whatever wrote the tables
        call()
    return chain(g.raw_cuda_graph())


def _set(kind, n, dt, driven=False, **kw):
    ham = W.tfim_chain(n, 1.0, 0.7) if kind == "tfim" else W.heisenberg_chain(n, np.full(n, 0.8))
    x, z, _ = hs.hs_parse_terms(ham.labels)
    if driven:
        return hs.hs_build_factors_td(x, z, ham.coeffs, 0.5 * np.asarray(ham.coeffs), n, 1.0, 4, 4, dt)
    return hs.hs_build_factors_masks(x, z, ham.coeffs, n, 1.0, 4, 4, dt, **kw)


@pytest.mark.parametrize("driven", [False, True])
@pytest.mark.parametrize("kind,method,dt", [("tfim", "FUSED", "c64"), ("tfim", "REG", "c64"), ("tfim", "REG", "c128"),
                                            ("heisenberg", "FUSED", "c128"), ("heisenberg", "AUTO", "c64")])
def test_sweeps(kind, method, dt, driven):
    n = 15  # (more than a tile: several sweeps)
    f = _set(kind, n, dt, driven)
    psi = torch.zeros(1 << n, dtype=torch.complex64 if dt == "c64" else torch.complex128, device="cuda")
    sweeps = _captured(lambda: hs.hs_evolve_ex(f, psi, 8, method=getattr(hs, "HS_METHOD_" + method)), psi)
    assert len(sweeps) >= 2
    assert all(kind == KERNEL for _, kind in sweeps)
    assert [edge == PROGRAMMATIC for edge, _ in sweeps] == [not driven] + [True] * (len(sweeps) - 1)


@pytest.mark.parametrize("driven", [False, True])
@pytest.mark.parametrize("method", [0, hs.HS_METHOD_REG])
def test_batch_levels(method, driven):
    jobs = [(_set("tfim", n, "c64", driven), torch.zeros(1 << n, dtype=torch.complex64, device="cuda"), 4)
            for n in (14, 15)]
    b = hs.hs_batch_create(jobs, method=method, use_graph=False)
    edges = [e for e, _ in _captured(lambda: hs.hs_batch_launch(b), jobs[0][1])]
    first = 2 if method == hs.HS_METHOD_REG else int(driven)  # (a register batch writes its tables first)
    assert len(edges) > first
    assert all(e != PROGRAMMATIC for e in edges[:first])
    assert all(e == PROGRAMMATIC for e in edges[first:])


def test_diagonals_built_late():
    n = 12
    g = torch.cuda.CUDAGraph(keep_graph=True)
    psi = torch.zeros(1 << n, dtype=torch.complex64, device="cuda")
    first = _set("tfim", n, "c64")
    hs.hs_evolve_ex(first, psi, 2, method=hs.HS_METHOD_FUSED)
    f = _set("tfim", n, "c64", defer_diagonals=True)
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        psi.mul_(1.0)
        hs.hs_evolve_ex(f, psi, 2, method=hs.HS_METHOD_FUSED)
    nodes = chain(g.raw_cuda_graph())
    at = [k for _, k in nodes].index(MEMSET)
    assert 0 < at < len(nodes) - 1  # behind the build, ahead of the sweeps
    assert all(e != PROGRAMMATIC for e, _ in nodes[:at + 1])


BUILD = """
import sys, os
import torch
sys.path[:0] = [{root!r}, {here!r}]
import test_gpu_launch_order as t
g = torch.cuda.CUDAGraph(keep_graph=True)
x = torch.zeros(4, device="cuda")
t._set("tfim", 12, "c64")
torch.cuda.synchronize()
s = torch.cuda.Stream()
with torch.cuda.graph(g, stream=s, capture_error_mode="relaxed"):
    x.mul_(1.0)
    f = t._set("tfim", 12, "c64")
print("KINDS", [k for _, k in t.chain(g.raw_cuda_graph())], flush=True)
os._exit(0)  # (the set's memory belongs to a graph that never ran)
"""


def test_a_build_ends_with_the_write():
    here = os.path.dirname(os.path.abspath(__file__))
    r = subprocess.run([sys.executable, "-c", BUILD.format(root=os.path.dirname(here), here=here)],
                       capture_output=True, text=True, timeout=300)
    line = [l for l in r.stdout.splitlines() if l.startswith("KINDS")]
    assert line, r.stderr[-2000:]
    kinds = eval(line[0][5:])
    assert kinds[-1] == MEMSET and KERNEL in kinds
