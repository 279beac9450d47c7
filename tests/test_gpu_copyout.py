"""The copy-out in bitstring order: one determinant, sizes around the sort's
tiles (4,096 pairs, 512 a warp), every bit of 64 spin-orbitals in use."""
import itertools

import numpy as np
import pytest

from paper_2411_07920_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_so,n_e,n", [(12, 4, 1), (28, 8, 511), (28, 8, 4096), (28, 8, 4097), (64, 6, 20_001), (40, 10, 70_000)])
def test_copy_out_is_sorted(n_so, n_e, n):
    from paper_2411_07920_gb300 import swcs
    rng = np.random.default_rng(n)
    w = I.small_case(n_so, n_e, 2, 5)
    strings = np.array([sum(1 << (2 * p) for p in s) for s in itertools.combinations(range(n_so // 2), n_e // 2)], np.uint64)
    pick = rng.choice(len(strings) ** 2, size=n, replace=False)  # in random order
    k = strings[pick // len(strings)] | (strings[pick % len(strings)] << np.uint64(1))
    a = rng.normal(size=n)
    with swcs.Context() as c:
        c.load_hamiltonian(w.h, w.g, n_so, n_e)
        c.set_state(k, a)
        ks, as_ = c.get_state()
        o = np.argsort(k)
        assert np.array_equal(ks, k[o]) and np.array_equal(as_, a[o])
        kg, sg = c.get_sigma()
        assert np.array_equal(kg, ks)
        assert np.abs(c.sigma_at(kg[:50]) - sg[:50]).max() < 1e-10
