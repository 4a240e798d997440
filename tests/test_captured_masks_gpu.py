"""A caller's graph of sweeps on the on-chip and cluster paths (whose draws are of
the sweeps it was captured for) replayed after a direct call that needs larger
mask buffers: the graph's buffers are still its own."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,layout,more", [(64, 0, 700), (296, 0, 300), (1008, 0, 200), (504, 1, 300)])
def test_replay_after_a_longer_call(L, layout, more):
    import torch
    import paper_1811_04384_gb300 as ising
    ising.load()
    seed, beta, n = 23 + L, 0.43, 20
    s = oracle.init_hot(L, seed)
    stream = torch.cuda.Stream()
    with ising.Lattice(L, seed, layout=layout, stream=stream) as lat:
        lat.set_clusters(0 if L == 64 else 1)
        assert lat.get_path() != ising.ISING_PATH_LAUNCHES
        lat.init_hot()
        lat.set_beta(beta)
        lat.sweep(n)
        lat.energy()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            lat.sweep(n)
        oracle.run(s, seed, beta, 0, n, n)
        t = 2 * n                                  # the captured call counts
        for _ in range(2):
            with torch.cuda.stream(stream):
                graph.replay()
            oracle.run(s, seed, beta, n, n, n)     # always the same sweeps
            lat.sweep(more)
            oracle.run(s, seed, beta, t, more, more)
            t += more
            more += 100
        np.testing.assert_array_equal(lat.get_spins(), s)
