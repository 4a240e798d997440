"""Several clusters through a series of calls: their pieces are numbered on from
call to call (one, two and four pieces, so that the agreement's two sets come in
either order), with other numbers of clusters and one between them, a call that
gives up at its first launch or a later one, and calls after it.  Against the
oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


# (clusters, sweeps, every, the launch that gives up or None): 24 and 6 sweeps are one piece, 70 two, 130 four
CALLS = [(2, 24, 4, None), (2, 70, 7, None), (2, 24, 1, None), (3, 130, 13, None), (1, 10, 5, None), (3, 6, 2, None),
         (2, 24, 3, 0), (2, 24, 3, None), (4, 130, 10, 2), (2, 6, 1, None), (2, 70, 5, None), (3, 6, 3, None)]


@pytest.mark.parametrize("L,layout", [(660, 0), (1008, 1)])
def test_series_of_calls(L, layout):
    import paper_1811_04384_gb300 as ising
    ising.load()
    seed, beta, t = 61 + L, 0.44, 0
    s = oracle.init_hot(L, seed)
    with ising.Lattice(L, seed, layout=layout) as lat:
        lat.init_hot()
        lat.set_beta(beta)
        for clusters, n, every, absent in CALLS:
            lat.set_clusters(clusters)
            if absent is not None:
                lat.inject_absent(absent)
            E, M = lat.sweep_record(n, every)
            Eo, Mo = oracle.run(s, seed, beta, t, n, every)
            t += n
            np.testing.assert_array_equal(E, Eo, err_msg=str((clusters, n, absent)))
            np.testing.assert_array_equal(M, Mo, err_msg=str((clusters, n, absent)))
        np.testing.assert_array_equal(lat.get_spins(), s)
