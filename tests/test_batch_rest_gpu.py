"""Calls of a batch whose sweeps are not whole chunks (short graphs run the
rest), chunks shorter than a short graph, uneven replicas, records in and out
of step; and lanes set twice before a sweep (the graphs hold the tile table)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

L, BETA, SEED = [64, 130, 32, 300], [0.3, 0.44, 0.5, 0.42], [5, 6, 7, 8]


def alone(ising, calls):
    out = []
    for r in range(len(L)):
        with ising.Lattice(L[r], SEED[r]) as lat:
            lat.init_hot()
            lat.set_beta(BETA[r])
            out.append([lat.sweep_record(int(n[r]), every) for n, every in calls] + [lat.get_spins()])
    return out


def check(ising, b, calls):
    got = [b.sweep(n, every=every) for n, every in calls]
    for r, want in enumerate(alone(ising, calls)):
        for (E, M), (Eo, Mo) in zip(got, want):
            np.testing.assert_array_equal(E[r], Eo)
            np.testing.assert_array_equal(M[r], Mo)
        np.testing.assert_array_equal(b.get_spins(r), want[-1])


@pytest.mark.parametrize("chunk", [50, 12, 7])
def test_rests(chunk):
    import paper_1811_04384_gb300 as ising
    ising.load()
    with ising.Batch(L, BETA, SEED, hot=[1] * 4) as b:
        b.set_tiling(128, chunk)
        check(ising, b, [([1, 0, 1, 1], 1), ([23, 9, 10, 11], 1), ([50, 50, 3, 49], 3), ([61, 12, 60, 1], 1),
                         ([99, 100, 101, 41], 7)])


def test_lanes_set_twice():
    import paper_1811_04384_gb300 as ising
    ising.load()
    with ising.Batch(L, BETA, SEED, hot=[1] * 4) as b:
        got = []
        for lanes in (4, 2, 4):
            b.set_lanes(lanes)
            if lanes == 2:
                continue                    # no sweep between: the graphs of four lanes are of another table
            got.append(b.sweep(13, every=1))
    for r, want in enumerate(alone(ising, [([13] * 4, 1), ([13] * 4, 1)])):
        for (E, M), (Eo, Mo) in zip(got, want):
            np.testing.assert_array_equal(E[r], Eo)
            np.testing.assert_array_equal(M[r], Mo)
