"""Register sweeps on pair rows: equal-coupling bonds, chunks of states, phases in shared slots.

Every case is checked against the FP64 oracle (complex128 max-abs 1e-12; complex64 max-abs
1e-5: the tolerances of the register sweep).  The Hamiltonians put XX, YY and ZZ of a pair
in every order, with equal coefficients (one BOND op), with one of the three different (value
table or single rotations), on neighbouring and distant qubits and on qubit 0 (the two halves
of a pair); state counts around the chunk size run a tile's phases for several states.
"""
import itertools

import numpy as np
import pytest

import oracle as O
from paper_2606_16959_gb300 import hs, workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_16959_gb300 import _build
    _build.build()
    O.build()
    hs.lib()


def _bonds(n, pairs, rng, spoil=None):
    labels, coeffs = [], []
    for k, (a, b) in enumerate(pairs):
        j = float(rng.uniform(-1.5, 1.5))
        for q, p in enumerate(list(itertools.permutations("XYZ"))[k % 6]):
            labels.append(W.label_of(n, {a: p, b: p}))
            coeffs.append(j * (1.25 if spoil == q else 1.0))
    return labels, coeffs


@pytest.mark.parametrize("dt", ["c64", "c128"])
@pytest.mark.parametrize("n,rhs,order", [(10, 1, 1), (13, 5, 1), (14, 4, 2), (16, 3, 4)])
@pytest.mark.parametrize("spoil", [None, 1])
def test_bonds_match_the_oracle(dt, n, rhs, order, spoil):
    rng = np.random.default_rng(100 * n + rhs)
    pairs = [(i, i + 1) for i in range(n - 1)] + [(n - 1, 0), (0, 5), (2, n - 2)]
    labels, coeffs = _bonds(n, pairs, rng, spoil)
    labels += [W.label_of(n, {q: "Z", (q + 3) % n: "Z"}) for q in range(n)] + [W.label_of(n, {q: "X"}) for q in range(n)]
    coeffs += list(rng.uniform(-1.0, 1.0, 2 * n))
    psi0 = np.stack([W.gaussian_state(n, rng) for _ in range(rhs)])
    x, z, _ = O.parse_terms(labels)
    want = (O.evolve_direct(x, z, np.asarray(coeffs), 0.7, 2, psi0) if order == 1 else
            O.evolve_direct_order(x, z, np.asarray(coeffs), 0.7, 2, psi0, order))
    tdt = torch.complex64 if dt == "c64" else torch.complex128
    for budget in (4, 8, 16):
        f = hs.hs_build_factors(labels, np.asarray(coeffs), 0.7, 2, budget, dt, order=order)
        for rb in ((5, 4) if dt == "c64" else (4,)):
            psi = torch.from_numpy(psi0).to("cuda", tdt)
            hs.hs_evolve_ex(f, psi, 2, method=hs.HS_METHOD_REG, reg_bits=rb)
            err = float(np.max(np.abs(psi.cpu().numpy().astype(np.complex128) - want)))
            assert err <= (1e-12 if dt == "c128" else 1e-5), (budget, rb, err)
        f.close()


@pytest.mark.parametrize("n,rhs", [(14, 1), (15, 2), (15, 4), (16, 7)])
def test_phase_factors_of_a_chunk(n, rhs):
    """Dense diagonal terms (every pair): patterns inside and across the register groups, more
    factors than a thread keeps for several states, and a tile's states one after another."""
    rng = np.random.default_rng(7 * n + rhs)
    labels, coeffs = [], []
    for _ in range(2):
        for a, b in itertools.combinations(range(n), 2):
            labels.append(W.label_of(n, {a: "Z", b: "Z"}))
        labels += [W.label_of(n, {q: "X"}) for q in range(n)]
    coeffs = rng.uniform(-1.0, 1.0, len(labels))
    psi0 = np.stack([W.gaussian_state(n, rng) for _ in range(rhs)])
    x, z, _ = O.parse_terms(labels)
    want = O.evolve_direct(x, z, coeffs, 0.5, 3, psi0)
    f = hs.hs_build_factors(labels, coeffs, 0.5, 3, 4, "c64")
    psi = torch.from_numpy(psi0).to("cuda", torch.complex64)
    hs.hs_evolve_ex(f, psi, 3, method=hs.HS_METHOD_REG)
    assert float(np.max(np.abs(psi.cpu().numpy().astype(np.complex128) - want))) <= 1e-5
    f.close()
