"""A batch of register sweeps gives its host descriptors back once its tables are on the device."""
import os

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


def _resident():
    with open("/proc/self/statm") as f:
        return int(f.read().split()[1]) * os.sysconf("SC_PAGE_SIZE")


def test_descriptors_are_freed():
    ham = W.heisenberg_chain(14, [1.0] * 14)
    f = hs.hs_build_factors(ham.labels, ham.coeffs, 1.0, 4, 4, "c64")
    psi = torch.zeros(4096, 1 << 14, dtype=torch.complex64, device="cuda")

    def batch(count):
        return hs.hs_batch_create([(f, psi[k], 4) for k in range(count)], method=hs.HS_METHOD_REG, use_graph=False)

    small = batch(64)
    hs.hs_batch_launch(small)
    torch.cuda.synchronize()
    big = batch(4096)  # two descriptors of some 20 KB a job and more
    before = _resident()
    hs.hs_batch_launch(big)
    torch.cuda.synchronize()
    hs.hs_batch_launch(big)
    torch.cuda.synchronize()
    assert before - _resident() > 4096 * 20000
    big.close()
    small.close()
