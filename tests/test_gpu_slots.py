"""Evolution with a propagator of known flip masks against the same matrix from its diagonals.

hs_spme keeps the masks of its result and hs_dia_evolve then works by slots (four steps or
more); the same values through hs_dia_create have no masks and take the diagonals.  Both sum
the same products in another order: tolerance 1e-13 sqrt(steps) relative for complex128 and
2e-6 sqrt(steps) for complex64 (sums of at most 300 products); values that are not finite
appear at the same rows.
"""
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


def _pair(n, dt, dtype, extra=()):
    ham = W.tfim_chain(n, 1.0, 0.3)
    labels = list(ham.labels) + [W.label_of(n, t) for t in extra]
    u, _, ok = hs.hs_spme(hs.hs_dia_from_terms(labels, np.append(ham.coeffs, [0.2] * len(extra))), dt)
    assert ok
    offs, diags = u.get()
    v = hs.hs_dia_create(n, {int(d): diags[int(d)] for d in offs}, "c128")
    if dtype == "c64":
        u, v = hs.hs_dia_convert(u, "c64"), hs.hs_dia_convert(v, "c64")
    return u, v


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n,rhs,steps", [(5, 1, 4), (6, 2, 5), (7, 3, 4), (8, 1, 9), (10, 5, 4), (11, 4, 3), (12, 1, 6), (13, 2, 4)])
def test_slots_match_diagonals(n, rhs, steps, dtype):
    # (a Y Y bond and an X Z term: masks of two flips and complex entries)
    u, v = _pair(n, 1e-3, dtype, ({0: "Y", n - 1: "Y"}, {1: "X", 2: "Z"}, {2: "Y"}))
    tdt = torch.complex64 if dtype == "c64" else torch.complex128
    psi = torch.from_numpy(np.stack([W.gaussian_state(n, np.random.default_rng(q)) for q in range(rhs)]))
    psi = psi.to("cuda", tdt)
    a, b = psi.clone(), psi.clone()
    hs.hs_dia_evolve(u, a, steps)
    hs.hs_dia_evolve(v, b, steps)
    tol = (2e-6 if dtype == "c64" else 1e-13) * np.sqrt(steps)
    assert float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b)) <= tol
    g = torch.cuda.CUDAGraph()
    c = psi.clone()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(g, stream=s):
        hs.hs_dia_evolve(u, c, steps)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(a, c)
    for bad in (float("inf"), float("nan")):
        a, b = psi.clone(), psi.clone()
        a[0, 3] = b[0, 3] = bad
        hs.hs_dia_evolve(u, a, 4)
        hs.hs_dia_evolve(v, b, 4)
        x, y = torch.view_as_real(a), torch.view_as_real(b)
        assert torch.equal(torch.isfinite(x), torch.isfinite(y))
        assert torch.equal(torch.isfinite(x[1:]).all(), torch.tensor(True, device="cuda"))


def test_overflow_on_the_way():
    """Values that overflow in complex64 after some steps: from there on the stored zeros count."""
    n = 8
    u, v = _pair(n, 1e-3, "c64")
    psi = torch.full((1, 1 << n), 3.0e38 + 3.0e38j, dtype=torch.complex64, device="cuda")
    a, b = psi.clone(), psi.clone()
    hs.hs_dia_evolve(u, a, 40)
    hs.hs_dia_evolve(v, b, 40)
    x, y = torch.view_as_real(a), torch.view_as_real(b)
    assert not bool(torch.isfinite(y).any()) and not bool(torch.isfinite(x).any())
