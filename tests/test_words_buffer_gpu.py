"""The buffer of the random-word chain's draws and plans is one for a handle's
life: a caller's graph captured after a call of one iteration runs more of them,
and stays good whatever the strips and sweeps of the calls between its replays."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,strips,others", [(84, 6, (42, 1, 2)), (504, 84, (252, 1, 12))])
def test_replays_among_direct_calls(L, strips, others):
    import torch
    import paper_1811_04384_gb300 as ising
    ising.load()
    seed, beta, t = 7 + L, 0.43, 0
    s = oracle.init_hot(L, seed)
    stream = torch.cuda.Stream()
    with ising.Lattice(L, seed, layout=ising.ISING_LAYOUT_COLUMN_INTERLEAVED, stream=stream) as lat:
        lat.init_hot()
        lat.set_beta(beta)
        lat.set_chain(ising.ISING_CHAIN_RANDOM_WORDS, strips)
        lat.sweep(1)
        oracle.rw_run(s, seed, beta, t, 1, strips, 1)
        t += 1
        lat.energy()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            lat.sweep(3)
        for other in others:
            with torch.cuda.stream(stream):
                graph.replay()
            oracle.rw_run(s, seed, beta, t, 3, strips, 3)
            t += 3
            lat.set_chain(ising.ISING_CHAIN_RANDOM_WORDS, other)
            lat.sweep(20 if L == 84 else 2)
            oracle.rw_run(s, seed, beta, t, 20 if L == 84 else 2, other, 1)
            t += 20 if L == 84 else 2
        np.testing.assert_array_equal(lat.get_spins(), s)
