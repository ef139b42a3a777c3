"""The two places above AUTO's complex128 line that stay with the staged sweeps, and their neighbours."""
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


# (terms, qubits, states, order, steps, register sweeps)
CASES = [
    ("tfim", 14, 6, 1, 3, False), ("tfim", 14, 7, 2, 2, False), ("tfim", 14, 8, 1, 3, True),
    ("tfim", 13, 12, 1, 3, True), ("tfim", 15, 3, 1, 3, True), ("chain", 14, 6, 1, 3, True),
    ("chain", 16, 2, 2, 1, False), ("chain", 16, 2, 2, 2, True), ("chain", 18, 1, 2, 1, False),
    ("chain", 15, 4, 2, 1, True), ("chain", 18, 2, 2, 1, True), ("chain", 17, 2, 1, 1, True),
    ("tfim", 17, 1, 2, 1, True),
]


@pytest.mark.parametrize("kind,n,rhs,order,steps,reg", CASES)
def test_lines(kind, n, rhs, order, steps, reg):
    ham = W.tfim_chain(n, 1.1, 0.7) if kind == "tfim" else W.heisenberg_chain(n, np.linspace(0.5, 1.5, n))
    f = hs.hs_build_factors(ham.labels, ham.coeffs, 1.0, 20, 4, "c128", order=order)
    plan = hs.hs_evolve_plan(f, rhs, steps)
    staged = hs.hs_evolve_plan(f, rhs, steps, method=hs.HS_METHOD_FUSED)
    assert plan == (hs.hs_evolve_plan(f, rhs, steps, method=hs.HS_METHOD_REG, tile_bits=10) if reg else staged)
    g = torch.Generator(device="cuda").manual_seed(n)
    psi = torch.randn(rhs, 1 << n, dtype=torch.complex128, device="cuda", generator=g)
    psi /= torch.linalg.vector_norm(psi, dim=1, keepdim=True)
    a, b = psi.clone(), psi.clone()
    hs.hs_evolve(f, a, steps)
    hs.hs_evolve_ex(f, b, steps, method=hs.HS_METHOD_FUSED)
    assert torch.equal(a, b) != reg
    assert float(torch.linalg.vector_norm(a - b, dim=1).max()) <= 1e-12
