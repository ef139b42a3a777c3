"""CPU checks that every register sweep the planner accepts fits a CTA's shared memory.

Sets with long diagonal runs have many classes of phase constants and several factor slots a
thread; in the largest tiles those and the tile do not fit in their first form.
"""
import numpy as np
import pytest

from paper_2606_16959_gb300 import hs

MOST = 227 * 1024


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2606_16959_gb300 import _build
    _build.build()
    hs.lib()


def dense(n, k, lo, hi, seed=None):
    """k diagonal terms on lo .. hi qubits each, then X on every qubit."""
    rng = np.random.default_rng(k if seed is None else seed)
    z = []
    while len(z) < k:
        m = sum(1 << int(i) for i in rng.choice(n, size=rng.integers(lo, hi + 1), replace=False))
        if m not in z:
            z.append(m)
    return [0] * k + [1 << i for i in range(n)], z + [0] * n, rng.uniform(0.1, 1.0, k + n)


# (dtype, tile bits, register bits, qubits, terms, fewest and most qubits of a term)
SETS = [
    ("c128", 13, 4, 16, 150, 3, 4), ("c128", 13, 4, 18, 150, 3, 4), ("c128", 13, 4, 16, 300, 3, 4),
    ("c128", 13, 4, 13, 60, 2, 2), ("c128", 13, 4, 13, 91, 1, 2), ("c128", 13, 4, 22, 300, 3, 4),
    ("c128", 13, 4, 13, 51, 2, 3), ("c128", 13, 4, 18, 74, 2, 3), ("c128", 12, 4, 20, 190, 2, 2),
    ("c128", 12, 4, 16, 300, 3, 4), ("c128", 9, 4, 22, 231, 2, 2), ("c64", 14, 5, 16, 150, 3, 4),
    ("c64", 14, 5, 20, 300, 3, 4), ("c64", 13, 5, 18, 300, 3, 4), ("c64", 13, 4, 20, 190, 2, 2),
    ("c64", 10, 5, 20, 300, 3, 4),
]


@pytest.mark.parametrize("dt,T,B,n,k,lo,hi", SETS)
def test_register_sweeps_fit(dt, T, B, n, k, lo, hi):
    x, z, c = dense(n, k, lo, hi)
    for driven in (False, True):
        for reserve in (0, 280, 12000):
            p = hs.hs_plan_register(x, z, c, n, 4, 3, T, B, dtype=dt, driven=driven, reserve=reserve)
            assert p["n_sweeps"] > 0 and p["n_plain"] == 0
            assert p["smem_max"] + reserve <= MOST


def test_higher_orders_fit():
    x, z, c = dense(14, 91, 2, 2)
    for order in (2, 4):
        p = hs.hs_plan_register(x, z, c, 14, 4, 2, 13, 4, order=order, dtype="c128")
        assert p["n_plain"] == 0 and p["smem_max"] <= MOST


def test_too_large_a_reserve_is_no_register_sweep():
    x, z, c = dense(13, 91, 1, 2)
    p = hs.hs_plan_register(x, z, c, 13, 4, 1, 13, 4, dtype="c128", reserve=100000)
    assert p["n_sweeps"] == 0 and p["n_plain"] > 0
