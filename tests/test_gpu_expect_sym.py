"""Expectation values of real symmetric matrices (H without odd numbers of Y) against dense sums.

hs_expectation takes a kernel of its own for them; the same H as a matrix uploaded with
hs_dia_create (nothing known about it) takes the general one.  Tolerance 1e-12 relative to
|H|_1 (FP64 sums of at most 2^13 x 60 products), and states that are not finite give what the
general kernel gives.
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


@pytest.mark.parametrize("dt", ["c64", "c128"])
@pytest.mark.parametrize("n,rhs", [(1, 1), (3, 2), (5, 3), (9, 4), (11, 5), (13, 7)])
def test_symmetric_expectation(dt, n, rhs):
    rng = np.random.default_rng(31 * n + rhs)
    terms = [{int(rng.integers(n)): "X"}, {0: "Z"}, {}]
    for _ in range(12):
        q = rng.choice(n, size=min(n, int(rng.integers(1, 5))), replace=False)
        terms.append({int(b): str(rng.choice(list("XYZ"))) for b in q})
    for odd in (False, True):  # without and with terms that have an odd number of Y
        use = [t for t in terms if odd or sum(p == "Y" for p in t.values()) % 2 == 0]
        labels, c = [W.label_of(n, t) for t in use], rng.uniform(-1, 1, len(use))
        H = hs.hs_dia_from_terms(labels, c)
        _, diags = H.get()
        G = hs.hs_dia_create(n, {d: diags[int(d)] for d in diags}, "c128")
        if dt == "c64":
            H, G = hs.hs_dia_convert(H, "c64"), hs.hs_dia_convert(G, "c64")
        psi = np.stack([W.gaussian_state(n, rng) for _ in range(rhs)])
        t = torch.from_numpy(psi).to("cuda", torch.complex64 if dt == "c64" else torch.complex128)
        v, nn = hs.hs_expectation(H, t)
        w, mm = hs.hs_expectation(G, t)
        scale = np.abs(c).sum()
        assert np.max(np.abs(v - w)) <= 1e-12 * scale and np.max(np.abs(nn - mm)) <= 1e-12
    t[0, 0] = float("inf")
    v, nn = hs.hs_expectation(H, t)
    w, mm = hs.hs_expectation(G, t)
    assert np.array_equal(np.isnan(v), np.isnan(w)) and np.array_equal(np.isfinite(nn), np.isfinite(mm))
