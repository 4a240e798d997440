"""What is left of a batch's call after whole chunks, in one more chunk or in
short graphs, on either side of the rule: the series are those of the default
chunk."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

L, BETA, SEED = [64, 130, 32], [0.3, 0.44, 0.5], [5, 6, 7]


@pytest.fixture(scope="module")
def ising():
    import paper_1811_04384_gb300 as p
    p.load()
    return p


def series(ising, chunk, calls):
    with ising.Batch(L, BETA, SEED, hot=[1] * 3) as b:
        if chunk:
            b.set_tiling(128, chunk)
        out = [x for n in calls for EM in b.sweep(n, every=2) for x in EM]
        return out + [b.get_spins(r) for r in range(3)] + [b.t(r) for r in range(3)]


@pytest.mark.parametrize("chunk,calls", [(50, [33, 34, 40, 83, 84, 90]), (200, [142, 143, 350]), (1024, [730, 731, 1000]),
                                         (12, [7, 11, 13]), (1, [3])])
def test_rule(ising, chunk, calls):
    for a, b in zip(series(ising, chunk, calls), series(ising, 0, calls)):
        np.testing.assert_array_equal(a, b)
