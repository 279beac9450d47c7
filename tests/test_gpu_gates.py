"""The in-place gate sequence and its tape, bit for bit against the oracle:
cluster and grid launches (up to 16,384 determinants and above), cuts that stay
in the counted band and cuts that leave it (large angles), partners put aside
and kept after all, ties, one kept determinant, the magnitude criterion, and the
backward pass over one tape and over replayed segments."""
import numpy as np
import pytest

import oracle as O
from paper_2411_07920_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TOL = 1e-10


@pytest.mark.parametrize("n_so,n_e,n_ops,seed,n_keep,eps,scale", [
    (12, 4, 12, 61, 6, 0.0, 1.0),
    (16, 6, 60, 7, 20, 0.0, 6.0),
    (20, 10, 150, 3, 1000, 0.0, 1.0),   # positions and index slots reused many times over
    (20, 10, 150, 3, 1000, 0.0, 6.0),
    (28, 8, 120, 5, 1, 0.0, 1.0),
    (28, 8, 120, 5, 7, 0.0, 6.0),
    (16, 6, 40, 9, 0, 1e-3, 1.0),
    (24, 8, 80, 73, 500, 1e-5, 5.0),
    (40, 10, 100, 3, 16384, 0.0, 1.0),  # the largest cluster launch
    (40, 10, 100, 3, 16385, 0.0, 1.0),  # the smallest grid launch
    (36, 10, 120, 4, 70_000, 0.0, 5.0),
])
@pytest.mark.parametrize("blocks", [0, 3])
def test_gates_bit_exact(n_so, n_e, n_ops, seed, n_keep, eps, scale, blocks):
    from paper_2411_07920_gb300 import swcs
    if blocks and n_keep > 2000:
        pytest.skip("small states only")
    w = I.small_case(n_so, n_e, n_ops, seed, n_keep=n_keep)
    th = w.theta * scale
    ko, ao = O.apply_ansatz(n_so, n_e, w.ops, th, n_keep, eps=eps)
    with swcs.Context() as c:
        c.load_hamiltonian(w.h, w.g, n_so, n_e)
        c.set_option("gate_blocks", blocks)
        c.set_truncation_threshold(eps)
        c.apply_ansatz(w.ops, th, n_keep)
        k, a = c.get_state()
        assert np.array_equal(k, ko) and np.array_equal(a, ao)
        half = n_ops // 2  # continued from a state
        c.apply_ansatz(w.ops[:half], th[:half], n_keep)
        c.apply_gates(w.ops[half:], th[half:], n_keep)
        k, a = c.get_state()
        assert np.array_equal(k, ko) and np.array_equal(a, ao)
        e1, d1 = c.energy_grad(w.ops, th, n_keep)
        k, a = c.get_state()
        assert np.array_equal(k, ko) and np.array_equal(a, ao)
        if len(ko) <= 1000:
            eo, do = O.energy_grad(n_so, n_e, w.h, w.g, w.ops, th, n_keep, eps=eps)
            assert abs(e1 - eo) < TOL and np.abs(d1 - do).max() < TOL


@pytest.mark.parametrize("n_keep,ckpt", [(3000, 7), (20_000, 20), (20_000, 1)])
def test_tape_in_segments(n_keep, ckpt):
    """A tape of 1 MiB does not hold all gates: the segments' derivatives are the whole tape's."""
    from paper_2411_07920_gb300 import swcs
    w = I.small_case(32, 8, 50, 11, n_keep=n_keep)
    with swcs.Context() as c:
        c.load_hamiltonian(w.h, w.g, w.n_so, w.n_e)
        e0, d0 = c.energy_grad(w.ops, w.theta, n_keep, ckpt)
        k0, a0 = c.get_state()
        c.set_option("adjoint_tape_mb", 1)
        e1, d1 = c.energy_grad(w.ops, w.theta, n_keep, ckpt)
        k1, a1 = c.get_state()
        assert abs(e0 - e1) < TOL and np.abs(d0 - d1).max() < TOL
        assert np.array_equal(k0, k1) and np.array_equal(a0, a1)


def test_zero_angles_keep_their_derivatives():
    """A new ADAPT operator at theta = 0: its partners have c = 0, stay in the projectors and leave the state."""
    from paper_2411_07920_gb300 import swcs
    w = I.small_case(16, 6, 20, 13)
    th = w.theta.copy()
    th[12:] = 0.0
    with swcs.Context() as c:
        c.load_hamiltonian(w.h, w.g, w.n_so, w.n_e)
        e, d = c.energy_grad(w.ops, th, 0)
        eo, do = O.energy_grad(16, 6, w.h, w.g, w.ops, th, 0)
        assert abs(e - eo) < TOL and np.abs(d - do).max() < TOL and np.abs(do[12:]).max() > 1e-4
        k, a = c.get_state()
        ko, ao = O.apply_ansatz(16, 6, w.ops, th, 0)
        assert np.array_equal(k, ko) and np.array_equal(a, ao)
