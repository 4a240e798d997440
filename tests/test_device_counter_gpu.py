"""The device's sweep counter: every path that advances it, followed by sweeps
that read it (graph replays), and a caller's own graph of sweeps, whose replays
the host does not see, followed by direct calls.  Against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

BETA = 0.43


@pytest.fixture(scope="module")
def ising():
    import paper_1811_04384_gb300 as p
    p.load()
    return p


# one warp, one band cluster, one cluster of two-word units, several clusters; the interleaved layout's
@pytest.mark.parametrize("L,layout,clusters", [(64, 0, 0), (128, 0, 0), (296, 0, 0), (1008, 0, 1), (1008, 0, 2),
                                               (84, 1, 0), (504, 1, 0), (1008, 1, 2)])
def test_on_chip_paths_then_graphs(ising, L, layout, clusters):
    seed = 3 + L
    with ising.Lattice(L, seed, layout=layout) as lat:
        lat.set_clusters(clusters)
        assert lat.get_path() != ising.ISING_PATH_LAUNCHES
        lat.init_hot()
        lat.set_beta(BETA)
        lat.sweep(3)
        lat.sweep_record(101, 50)              # more than one piece
        lat.set_path(ising.ISING_PATH_LAUNCHES)
        E, M = lat.sweep_record(35, 1)
        S, t = lat.get_spins(), lat.t
    s = oracle.init_hot(L, seed)
    oracle.run(s, seed, BETA, 0, 104, 104)
    Eo, Mo = oracle.run(s, seed, BETA, 104, 35, 1)
    np.testing.assert_array_equal(E, Eo)
    np.testing.assert_array_equal(M, Mo)
    np.testing.assert_array_equal(S, s)
    assert t == 139


def test_states_then_graphs(ising):
    L, seed = 1000, 8
    rng = np.random.default_rng(2)
    states = [np.where(rng.random((L, L)) < 0.5, 1, -1).astype(np.int8) for _ in range(3)]
    with ising.Lattice(L, seed) as lat:
        lat.set_path(ising.ISING_PATH_LAUNCHES)
        lat.set_beta(BETA)
        lat.run_states(states, 4, 2)
        E, M = lat.sweep_record(33, 1)
        S = lat.get_spins()
    s = states[2].copy()
    oracle.run(s, seed, BETA, 8, 4, 4)
    Eo, Mo = oracle.run(s, seed, BETA, 12, 33, 1)
    np.testing.assert_array_equal(E, Eo)
    np.testing.assert_array_equal(M, Mo)
    np.testing.assert_array_equal(S, s)


# a side whose chunks are graphs of the library's own (the rest of a call is not) and one without
@pytest.mark.parametrize("L", [130, 2400])
@pytest.mark.parametrize("replays", [0, 1, 3])
@pytest.mark.parametrize("after", ["sweep", "record", "states"])
def test_replays_then_direct_calls(ising, L, replays, after):
    import torch
    seed, n = 19, 34 if L == 130 else 4
    stream = torch.cuda.Stream()
    with ising.Lattice(L, seed, stream=stream) as lat:
        lat.set_path(ising.ISING_PATH_LAUNCHES)
        lat.init_hot()
        lat.set_beta(BETA)
        lat.sweep(2)
        lat.energy()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            lat.sweep(3)
        with torch.cuda.stream(stream):
            for _ in range(replays):
                graph.replay()
        t = 2 + 3 * replays
        s = oracle.init_hot(L, seed)
        oracle.run(s, seed, BETA, 0, t, t)
        if after == "states":
            E, M = (x[0] for x in lat.run_states([s], n, 1))
        elif after == "record":
            E, M = lat.sweep_record(n, 1)
        else:
            lat.sweep(n)
        S = lat.get_spins()
    Eo, Mo = oracle.run(s, seed, BETA, t, n, 1)
    if after != "sweep":
        np.testing.assert_array_equal(E, Eo)
        np.testing.assert_array_equal(M, Mo)
    np.testing.assert_array_equal(S, s)
