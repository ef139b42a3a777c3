"""Which kernel an evolution of a Taylor propagator runs, and its switch to the stored diagonals.

Once an amplitude is not finite the stored zeros count (0 times infinity): the rows it reaches in
one step are those of all stored diagonals, more than those of the flip masks.  The state starts
with one amplitude whose phase turns past the largest complex64 value after some twenty steps.
"""
import numpy as np
import pytest

from paper_2606_16959_gb300 import hs
from test_gpu_slots import _pair

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_16959_gb300 import _build
    _build.build()
    hs.lib()


def _launches(m, psi, steps):
    before = hs.hs_kernel_launches()
    hs.hs_dia_evolve(m, psi, steps)
    return hs.hs_kernel_launches() - before


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n,steps,slots", [(5, 8, False), (6, 4, True), (9, 3, False), (10, 4, True), (13, 9, True)])
def test_which_kernel_runs(n, steps, slots, dtype):
    u, v = _pair(n, 1e-3, dtype)
    psi = torch.zeros(1 << n, dtype=torch.complex64 if dtype == "c64" else torch.complex128, device="cuda")
    assert _launches(v, psi, steps) == steps
    assert _launches(u, psi, steps) == steps + (1 if slots else 0)  # (the gather)


def test_switch_after_an_overflow():
    n = 10
    u, v = _pair(n, 1e-3, "c64")
    seen = 0
    # (not row 0: the kernel of the diagonals multiplies amplitude 0 by zero for the rows outside
    # a diagonal, and so spreads it to every row)
    for row in (341, 700):
        for steps in range(8, 40):
            a = torch.zeros(1 << n, dtype=torch.complex64, device="cuda")
            a[row] = 3.0e38 + 3.0e38j
            b = a.clone()
            hs.hs_dia_evolve(u, a, steps)
            hs.hs_dia_evolve(v, b, steps)
            x, y = (~torch.isfinite(torch.view_as_real(s)) for s in (a, b))
            assert torch.equal(x, y)
            bad = int(y.any(dim=1).sum())
            seen += 1 < bad < 1 << n
    assert seen > 0
