"""Energy, sigma_D-based gradients and the pool sweep from the pairs of the
state's determinants (options "energy" 0 and "pairs" 1) against the oracle and
against the row sweep: orbital counts at the edges of the kernels' layouts (16
and 17 spatial orbitals, 32), two electrons of a spin (no same-spin triples),
more electrons than holes, one determinant, states whose groups cross the
32-determinant items, and determinants without any order or connection."""
import numpy as np
import pytest

import oracle as O
from paper_2411_07920_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TOL = 1e-10  # the path's tolerance against the oracle


def _check(c, w, k, a, mode="both"):
    e0, n0 = O.energy(w.n_so, w.h, w.g, k, a)
    e, n2 = c.energy()
    assert abs(e - e0) < TOL and abs(n2 - n0) < TOL * max(1.0, n0)
    c.set_option("pairs", 1)
    g = c.pool_gradients()
    es, n2s = c.sweep_energy()
    c.set_option("pairs", -1)
    go = O.pool_gradients(w.n_so, w.h, w.g, k, a)
    assert np.abs(g - go).max() < TOL
    assert abs(es - e0) < TOL and abs(n2s - n0) < TOL * max(1.0, n0)


@pytest.mark.parametrize("n_so,n_e,n_ops,n_keep", [
    (6, 4, 8, 0),        # three spatial orbitals: a single triple
    (8, 4, 12, 0),       # two electrons of a spin: no same-spin triple is occupied
    (8, 6, 12, 0),
    (10, 8, 20, 0),      # one hole per spin
    (12, 4, 10, 0),
    (22, 8, 40, 333),
    (32, 6, 40, 300),    # 16 spatial orbitals: two uses of an element share a warp
    (34, 6, 40, 300),    # 17: they do not
    (30, 20, 25, 150),   # more electrons than holes
    (52, 12, 40, 200),
    (64, 6, 40, 250),    # 32 spatial orbitals
])
def test_pairs_against_oracle(n_so, n_e, n_ops, n_keep):
    from paper_2411_07920_gb300 import swcs
    w = I.small_case(n_so, n_e, n_ops, 17, n_keep=n_keep)
    with swcs.Context() as c:
        c.load_hamiltonian(w.h, w.g, n_so, n_e)
        c.apply_ansatz(w.ops, w.theta, n_keep)
        k, a = c.get_state()
        _check(c, w, k, a)
        ed, d = c.energy_grad(w.ops, w.theta, n_keep)
        eo, do = O.energy_grad(n_so, n_e, w.h, w.g, w.ops, w.theta, n_keep)
        assert abs(ed - eo) < TOL and np.abs(d - do).max() < TOL


@pytest.mark.parametrize("n_so,n_e,n", [(12, 6, 1), (12, 6, 400), (14, 6, 700), (28, 8, 33), (28, 8, 500)])
def test_pairs_arbitrary_states(n_so, n_e, n):
    """Determinants drawn over the whole sector: 1, a full 12/6 sector (20 x 20), crowded groups, few connections."""
    import itertools

    from paper_2411_07920_gb300 import swcs
    rng = np.random.default_rng(n_so * 1000 + n)
    w = I.small_case(n_so, n_e, 4, 5)
    strings = [sum(1 << (2 * p) for p in s) for s in itertools.combinations(range(n_so // 2), n_e // 2)]
    pick = rng.choice(len(strings) ** 2, size=n, replace=False)
    k = np.sort(np.array([strings[i // len(strings)] | (strings[i % len(strings)] << 1) for i in pick], np.uint64))
    a = rng.normal(size=n)
    with swcs.Context() as c:
        c.load_hamiltonian(w.h, w.g, n_so, n_e)
        c.set_state(k, a)
        _check(c, w, k, a)


def test_pairs_agree_with_rows_and_subset():
    """A larger state: both sweeps, the subset form, and an untouched entry outside the subset."""
    import torch

    from paper_2411_07920_gb300 import swcs
    w = I.small_case(40, 10, 80, 23, n_keep=20_000)
    with swcs.Context() as c:
        c.load_hamiltonian(w.h, w.g, w.n_so, w.n_e)
        c.apply_ansatz(w.ops, w.theta, 20_000)
        out = []
        for pairs in (0, 1):
            c.set_option("pairs", pairs)
            out.append((c.pool_gradients(), c.sweep_energy()))
        assert np.abs(out[0][0] - out[1][0]).max() < TOL
        assert abs(out[0][1][0] - out[1][1][0]) < TOL
        sub = torch.arange(3, c.pool_size(), 7, dtype=torch.int64, device="cuda")
        g = torch.full((c.pool_size(),), 7.0, dtype=torch.float64, device="cuda")
        c.pool_gradients_dev(g, sub)
        g = g.cpu().numpy()
        s = sub.cpu().numpy()
        assert np.abs(g[s] - out[0][0][s]).max() < TOL
        rest = np.ones(len(g), bool)
        rest[s] = False
        assert (g[rest] == 7.0).all()


def test_pairs_do_not_apply():
    """One electron of each spin: no three-body matrix; the option leaves the row sweep in place."""
    from paper_2411_07920_gb300 import swcs
    w = I.small_case(12, 2, 6, 3)
    with swcs.Context() as c:
        c.load_hamiltonian(w.h, w.g, 12, 2)
        c.apply_ansatz(w.ops, w.theta, 0)
        k, a = c.get_state()
        _check(c, w, k, a)
