"""The launch path of the column-interleaved layout with a half-sweep split over
the four warps of a block (fields and rows), on either side of its limit: sides
whose last block of columns is part empty, records and none, in graphs and
outside, both schemes, thresholds of 2^32 and 0; against the oracle, or for larger
sides the cluster path's dense form."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ising():
    import paper_1811_04384_gb300 as p
    p.load()
    return p


def series(ising, L, path, beta, n, every, rng=0):
    with ising.Lattice(L, 0x0abc000000000000 + L, layout=ising.ISING_LAYOUT_COLUMN_INTERLEAVED) as lat:
        lat.set_path(path)
        lat.set_rng(rng)
        lat.init_hot()
        lat.set_beta(beta)
        lat.t = 2**32 - 7
        lat.sweep(3)
        E, M = lat.sweep_record(n, every)
        return E, M, lat.get_spins(), lat.energy(), lat.magnetization()


@pytest.mark.parametrize("L", [84, 168, 252, 336])
@pytest.mark.parametrize("beta", [0.0, 0.44, 4.0])
@pytest.mark.parametrize("rounds", [10, 7])
def test_against_oracle(ising, L, beta, rounds):
    seed, n, every = 0x0abc000000000000 + L, 37, 3             # a graph of ten records, and sweeps outside it
    E, M, S, e, m = series(ising, L, ising.ISING_PATH_LAUNCHES, beta, n, every,
                           ising.ISING_RNG_PHILOX4X32_7 if rounds == 7 else ising.ISING_RNG_PHILOX4X32_10)
    with oracle.sweep_rounds(rounds):
        s = oracle.init_hot(L, seed)
        oracle.run(s, seed, beta, 2**32 - 7, 3, 3)
        Eo, Mo = oracle.run(s, seed, beta, 2**32 - 4, n, every)
    np.testing.assert_array_equal(E, Eo)
    np.testing.assert_array_equal(M, Mo)
    np.testing.assert_array_equal(S, s)
    assert (e, m) == (oracle.energy(s), oracle.magnetization(s))


@pytest.mark.parametrize("L", [420, 1008, 1428, 1512, 1596])
def test_against_cluster_path(ising, L):
    a = series(ising, L, ising.ISING_PATH_LAUNCHES, 0.43, 35, 1)
    for x, y in zip(a, series(ising, L, ising.ISING_PATH_CLUSTER, 0.43, 35, 1)):
        np.testing.assert_array_equal(x, y)
