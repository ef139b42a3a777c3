"""A batch of register sweeps gives bitwise what its jobs give alone, also where a sweep has more
operations than a warp has lanes (its scale is a product over all of them)."""
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


def _ham(kind, n, rng):
    if kind == "bonds":
        return W.heisenberg_chain(n, rng.uniform(0.5, 1.5, size=n))
    if kind == "field":  # X rotations with tangents and cosines of their own
        labels = [W.label_of(n, {i: "X"}) for i in range(n)] + [W.label_of(n, {i: "Z", (i + 1) % n: "Z"}) for i in range(n)]
        return W.Hamiltonian("tfim", n, labels, rng.uniform(0.2, 1.5, size=2 * n))
    return W.tfim_chain(n, rng.uniform(0.5, 1.5), rng.uniform(0.5, 1.5))


@pytest.mark.parametrize("dt", ["c128", "c64"])
@pytest.mark.parametrize("kind", ["bonds", "field", "tfim"])
def test_batch_bitwise_alone(kind, dt):
    tdt = torch.complex64 if dt == "c64" else torch.complex128
    jobs, alone, most = [], [], 0
    for seed in range(12):
        rng = np.random.default_rng(seed)
        n = 10 + seed % 3
        ham = _ham(kind, n, rng)
        x, z, _ = hs.hs_parse_terms(ham.labels)
        most = max(most, hs.hs_plan_register(x, z, ham.coeffs, n, 8, 12, dtype=dt)["ops_max"])
        f = hs.hs_build_factors(ham.labels, ham.coeffs, 1.0, 12, 8, dt)
        g = torch.Generator(device="cuda").manual_seed(seed)
        psi = torch.randn(1 << n, dtype=tdt, device="cuda", generator=g)
        jobs.append((f, psi, 12))
        a = psi.clone()
        hs.hs_evolve_ex(f, a, 12, method=hs.HS_METHOD_REG)
        alone.append(a)
    assert most > 32
    b = hs.hs_batch_create(jobs, method=hs.HS_METHOD_REG)
    assert b.n_separate == 0
    hs.hs_batch_launch(b)
    for (_, psi, _), a in zip(jobs, alone):
        assert torch.equal(psi, a)
    b.close()
