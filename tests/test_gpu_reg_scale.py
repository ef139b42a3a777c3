"""The scale of complex64 register sweeps of bonds is applied unrounded.

A bond leaves its phase e^{-i theta} in the sweep's complex scale.  Rounded to complex64 the
scale would shift the norm by up to 6e-8 a sweep, the same way at every repeated sweep.  The
angles here are such that this shift is 1.24e-5 and 1.23e-5 over the 420 sweeps of 300 steps
(12 bonds in 300 of them, 10 in 120), while the other roundings that move the norm one way (that
of w, and the norm of the forms a bond stands for) stay below 1.5e-6 together.
"""
import numpy as np
import pytest

from paper_2606_16959_gb300 import hs, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N, STEPS = 16, 300


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_16959_gb300 import _build
    _build.build()
    hs.lib()


def _norm(psi):
    return float(torch.linalg.vector_norm(psi.to(torch.complex128)))


# budget 4: one bond to a factor; 16: two
@pytest.mark.parametrize("budget,theta", [(4, 0.014302716593413811), (16, 0.011440856643230312)])
@pytest.mark.parametrize("how", ["evolve", "evolve 4 bits", "batch"])
def test_norm_of_many_steps(how, budget, theta):
    ham = W.heisenberg_chain(N, np.full(N, theta * STEPS))
    f = hs.hs_build_factors(ham.labels, ham.coeffs, 1.0, STEPS, budget, "c64")
    g = torch.Generator(device="cuda").manual_seed(7)
    psi = torch.randn(1 << N, dtype=torch.complex64, device="cuda", generator=g)
    psi /= torch.linalg.vector_norm(psi)
    before = _norm(psi)
    if how == "batch":
        b = hs.hs_batch_create([(f, psi, STEPS)], method=hs.HS_METHOD_REG)
        hs.hs_batch_launch(b)
    else:
        hs.hs_evolve_ex(f, psi, STEPS, method=hs.HS_METHOD_REG, reg_bits=4 if "4" in how else 5)
    assert abs(_norm(psi) / before - 1.0) <= 3e-6
