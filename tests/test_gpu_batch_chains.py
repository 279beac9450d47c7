"""The batch's density-matrix sweeps: chains of launches after the persistent kernel, for the instances whose sweep
the single context would take through the density matrices."""
import numpy as np
import pytest

from paper_2411_07920_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TOL = 1e-10


@pytest.fixture(scope="module")
def S():
    from paper_2411_07920_gb300 import swcs
    return swcs


@pytest.mark.parametrize("lanes", [1, 6])
def test_batch_density_matrix_chains(S, lanes):
    """Instances whose sweep runs through the density matrices after the persistent kernel (34/12 states of some
    thousand determinants; six of them make chains of two and one), beside one whose rows stay inside it: energies,
    norms and gradients of the single context's row sweep, twice from one graph, and the state is the same."""
    ws = [I.small_case(34, 12, 40, 300 + k, n_keep=2000 + 500 * k) for k in range(lanes)]
    ws.append(I.small_case(16, 6, 25, 320, n_keep=120))
    b = S.Batch()
    for w in ws:
        b.add(w.h, w.g, w.n_so, w.n_e, w.ops, w.theta, w.n_keep)
    b.build(autotune=False)
    ref = []
    for w in ws:
        ctx = S.Context()
        ctx.set_option("pairs", 0)
        ctx.set_option("sweep", 2)
        ctx.load_hamiltonian(w.h, w.g, w.n_so, w.n_e)
        ctx.apply_ansatz(w.ops, w.theta, w.n_keep)
        g = ctx.pool_gradients()
        ref.append((*ctx.sweep_energy(), g))
        ctx.close()
    for rep in range(2):
        b.run()
        for i in range(len(ws)):
            e, n2, g = b.results(i)
            assert abs(e - ref[i][0]) < TOL and abs(n2 - ref[i][1]) < 1e-13, i
            assert np.abs(g - ref[i][2]).max() < TOL, i
    b.close()
