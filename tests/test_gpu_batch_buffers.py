"""The batch's graph holds its instances' buffers by address: a back-to-back run between two launches of the graph
must leave those in place."""
import numpy as np
import pytest

from paper_2411_07920_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [0, 1])
def test_graph_runs_again_after_back_to_back(mode):
    from paper_2411_07920_gb300 import swcs as S
    ws = [I.small_case(16, 6, 25, 202, n_keep=120), I.small_case(24, 8, 35, 206, n_keep=600)]
    b = S.Batch()
    for w in ws:
        b.add(w.h, w.g, w.n_so, w.n_e, w.ops, w.theta, w.n_keep)
    b.set_tuning(mode, 4096, 2, 2)
    b.build(autotune=False)
    got = []
    for run in (b.run, b.run_serial, b.run):
        run()
        got.append([b.results(i) for i in range(len(ws))])
    for r in got[1:]:
        for (e, n2, g), (e0, n20, g0) in zip(r, got[0]):
            assert abs(e - e0) < 1e-10 and abs(n2 - n20) < 1e-13
            assert np.abs(g - g0).max() < 1e-10
    b.close()
