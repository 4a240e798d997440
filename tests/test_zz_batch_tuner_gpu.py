"""The batch tuner times the graphs of the chunk it is about to choose, not their
capture nor the short graphs of a call's rest: for small replicas, whose graphs
cost the host as much as the GPU, chunks of ten sweeps take a fifth longer."""
import pytest

pytestmark = pytest.mark.gpu


# 40 graphs of 10 sweeps, or less than one of 50: a whole chunk of any candidate either way
@pytest.mark.parametrize("sweeps", [400, 20])
def test_small_replicas_take_long_chunks(sweeps):
    import paper_1811_04384_gb300 as ising
    from paper_1811_04384_gb300 import tuning
    ising.load()
    best = tuning.tune_batch([64] * 4, [0.44] * 4, [1, 2, 3, 4], [1] * 4, sweeps=sweeps)
    assert best["graph_chunk"] in (50, 200)
