"""Register sweeps whose tables take much shared memory: long diagonal runs in large tiles.

Their phase factors and class constants are kept in one of three forms (slots of their own,
shared slots, local memory); the arithmetic is the same.  Tolerances against the FP64 oracle:
complex128 1e-12 max-abs, complex64 1e-5 max-abs (as for every register sweep); a batch is
bitwise what its jobs are alone.
"""
import numpy as np
import pytest

import oracle as O
from paper_2606_16959_gb300 import hs, workloads as W
from test_register_plan_host import dense

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

REG = hs.HS_METHOD_REG


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_16959_gb300 import _build
    _build.build()
    O.build()
    hs.lib()


def _tdt(dt):
    return torch.complex64 if dt == "c64" else torch.complex128


# (dtype, tile bits, register bits, qubits, terms, fewest and most qubits of a term, some sweep is lean)
SETS = [
    ("c128", 13, 4, 13, 60, 2, 2, True), ("c128", 13, 4, 14, 150, 3, 4, True), ("c128", 13, 4, 16, 150, 3, 4, True),
    ("c128", 13, 4, 14, 56, 3, 3, False), ("c128", 12, 4, 14, 150, 3, 4, True), ("c64", 14, 5, 16, 150, 3, 4, False),
    ("c64", 13, 4, 16, 300, 3, 4, None), ("c64", 13, 5, 16, 300, 3, 4, None),
]


@pytest.mark.parametrize("dt,T,B,n,k,lo,hi,lean", SETS)
def test_matches_oracle(dt, T, B, n, k, lo, hi, lean):
    x, z, c = dense(n, k, lo, hi)
    c = c * 0.1
    p = hs.hs_plan_register(x, z, c, n, 4, 2, T, B, dtype=dt)
    assert p["n_plain"] == 0 and (lean is None or (p["n_lean"] > 0) == lean)
    rng = np.random.default_rng(n)
    psi0 = np.stack([W.gaussian_state(n, rng) for _ in range(2)])
    f = hs.hs_build_factors_masks(x, z, c, n, 0.5, 2, 4, dt)
    psi = torch.from_numpy(psi0).to("cuda", _tdt(dt))
    hs.hs_evolve_ex(f, psi, 2, method=REG, tile_bits=T, reg_bits=B)
    got = psi.cpu().numpy()
    xa, za = np.array(x, dtype=np.uint64), np.array(z, dtype=np.uint64)
    for r in range(2):
        want = O.evolve_direct(xa, za, c, 0.5, 2, psi0[r])
        assert np.max(np.abs(got[r] - want)) <= (1e-12 if dt == "c128" else 1e-5)


def test_driven_matches_oracle():
    n = 13
    x, z, c = dense(n, 60, 2, 2)
    a, b = np.where(np.arange(len(c)) < 60, 0.0, c), np.where(np.arange(len(c)) < 60, c, 0.0)
    drive = np.array([0.2, 0.5, 0.9])
    psi0 = W.gaussian_state(n, np.random.default_rng(3))
    f = hs.hs_build_factors_td(x, z, a, b, n, 0.6, 3, 4, "c128")
    psi = torch.from_numpy(psi0).to("cuda")
    hs.hs_evolve_td(f, psi, drive, method=REG, tile_bits=13)
    xa, za = np.array(x, dtype=np.uint64), np.array(z, dtype=np.uint64)
    want = O.evolve_direct_td(xa, za, a, b, drive, 0.6, psi0)
    assert np.max(np.abs(psi.cpu().numpy() - want)) <= 1e-12


# The header and prefix table of a batch leave less room than a launch of its own has: the first three
# sets then take another form than alone.
@pytest.mark.parametrize("dt,T,B,n,k,lo,hi", [("c128", 13, 4, 14, 56, 3, 3), ("c128", 13, 4, 13, 51, 2, 3),
                                              ("c128", 13, 4, 14, 114, 3, 3), ("c64", 13, 5, 16, 300, 3, 4)])
def test_batch_is_bitwise(dt, T, B, n, k, lo, hi):
    x, z, c = dense(n, k, lo, hi)
    f = hs.hs_build_factors_masks(x, z, c, n, 0.5, 3, 4, dt)
    g = torch.Generator(device="cuda").manual_seed(k)
    states = [torch.randn(1 << n, dtype=_tdt(dt), device="cuda", generator=g) for _ in range(3)]
    alone = [s.clone() for s in states]
    for s in alone:
        hs.hs_evolve_ex(f, s, 3, method=REG, tile_bits=T, reg_bits=B)
    b = hs.hs_batch_create([(f, s, 3) for s in states], method=REG, tile_bits=T, reg_bits=B)
    assert b.n_separate == 0
    hs.hs_batch_launch(b)
    for s, r in zip(states, alone):
        assert torch.equal(s, r)
    b.close()
