"""The launch path on either side of the side up to which it replays graphs
(32,768 thread items): records over several replays and a rest, sweeps without
records, ragged sides, both layouts; and a call that several clusters give up
between its pieces, which goes on there.  Against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ising():
    import paper_1811_04384_gb300 as p
    p.load()
    return p


# 585 x 56 = 32,760 items and 586 x 56 = 32,816; interleaved 567 x 54 and 588 x 56
CASES = [(2338, 0), (2340, 0), (2342, 0), (2268, 1), (2352, 1)]


def test_limit(ising):
    got, jobs = [], []
    for L, layout in CASES:
        with ising.Lattice(L, L + 5, layout=layout) as lat:
            lat.set_path(ising.ISING_PATH_LAUNCHES)
            lat.init_hot()
            lat.set_beta(0.43)
            lat.sweep(33)                          # a graph, and one outside
            E, M = lat.sweep_record(71, 3)         # two graphs of ten records, three outside, two sweeps
            got.append((E, M, lat.get_spins(), lat.t))
        jobs.append((L, L + 5, 0.43, True, 104, 1))
    for (E, M, S, t), (Eo, Mo, So), case in zip(got, oracle.run_jobs(jobs), CASES):
        at = np.arange(33 + 3, 33 + 72, 3) - 1
        np.testing.assert_array_equal(E, Eo[at], err_msg=str(case))
        np.testing.assert_array_equal(M, Mo[at], err_msg=str(case))
        np.testing.assert_array_equal(S, So, err_msg=str(case))
        assert t == 104


# four pieces of 45 sweeps: the second launch writes nothing, 135 sweeps on the launch path
@pytest.mark.parametrize("layout,clusters,every", [(0, 2, 7), (0, 4, 45), (1, 2, 5), (1, 3, 1)])
def test_pieces_given_up(ising, layout, clusters, every):
    L, seed, n = 1008, 1011, 180
    with ising.Lattice(L, seed, layout=layout) as lat:
        lat.set_clusters(clusters)
        assert lat.get_path() == ising.ISING_PATH_CLUSTER
        lat.init_hot()
        lat.set_beta(0.43)
        lat.inject_absent(1)
        E, M = lat.sweep_record(n, every)
        E2, M2 = lat.sweep_record(3, 1)
        S = lat.get_spins()
    s = oracle.init_hot(L, seed)
    Eo, Mo = oracle.run(s, seed, 0.43, 0, n, every)
    Eo2, Mo2 = oracle.run(s, seed, 0.43, n, 3, 1)
    for a, b in ((E, Eo), (M, Mo), (E2, Eo2), (M2, Mo2), (S, s)):
        np.testing.assert_array_equal(a, b)
