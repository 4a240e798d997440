"""The fused half-sweep's strips of word columns: one strip, strips of unequal
width, one-word strips, ragged row groups, block shapes whose last block is
part empty, single lattice and batch, against the oracle bit for bit."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ising():
    import paper_1811_04384_gb300 as p
    p.load()
    return p


# L: words per row W = ceil(L / 42): 1, 2, 31, 32 (one strip), 33 (17 + 16), 65 (22 + 22 + 21)
@pytest.mark.parametrize("L,bw,bg", [(4, 0, 64), (42, 0, 128), (46, 16, 2), (1302, 0, 256), (1344, 0, 128),
                                     (1346, 0, 192), (1346, 32, 1), (1346, 64, 4), (2694, 0, 128), (2730, 16, 8)])
@pytest.mark.parametrize("beta", [0.0, 1 / 2.269])
def test_strips_lattice(ising, L, bw, bg, beta):
    seed = 0x1234567800000000 + L
    with ising.Lattice(L, seed) as lat:
        lat.set_path(ising.ISING_PATH_LAUNCHES)
        lat.set_item_lanes(1)
        lat.set_tiling(4, bw, bg)
        lat.init_hot()
        lat.set_beta(beta)
        lat.t = 2**32 - 2                      # the counter's high word changes on the way
        E, M = lat.sweep_record(3, 1)
        spins = lat.get_spins()
    s = oracle.init_hot(L, seed)
    Eo, Mo = oracle.run(s, seed, beta, 2**32 - 2, 3, 1)
    np.testing.assert_array_equal(E, Eo)
    np.testing.assert_array_equal(M, Mo)
    np.testing.assert_array_equal(spins, s)


@pytest.mark.parametrize("threads", [64, 128, 256])
def test_strips_batch(ising, threads):
    L = [6, 42, 44, 1346, 1302, 90]
    beta = [0.0, 0.3, 0.44, 0.44, 2.9, 0.6]
    seed = [3 + k for k in range(len(L))]
    with ising.Batch(L, beta, seed, hot=[1] * len(L)) as b:
        b.set_tiling(threads, 2)
        E, M = b.sweep(3, every=1)
        spins = [b.get_spins(r) for r in range(len(L))]
    for r in range(len(L)):
        s = oracle.init_hot(L[r], seed[r])
        Eo, Mo = oracle.run(s, seed[r], beta[r], 0, 3, 1)
        np.testing.assert_array_equal(E[r], Eo)
        np.testing.assert_array_equal(M[r], Mo)
        np.testing.assert_array_equal(spins[r], s)


# word row groups N / 4 = 1, 4, 5 in blocks of 4; column pairs 42, 168, 210 in blocks of 32
@pytest.mark.parametrize("L", [84, 336, 420])
@pytest.mark.parametrize("rng,rounds", [(0, 10), (1, 7)])
@pytest.mark.parametrize("path", [1, 3])
def test_interleaved_row_keys(ising, L, rng, rounds, path):
    seed = 0xabcdef0000000011 + L
    with ising.Lattice(L, seed, layout=ising.ISING_LAYOUT_COLUMN_INTERLEAVED) as lat:
        lat.set_path(path)
        lat.set_rng(rng)
        lat.init_hot()
        lat.set_beta(0.43)
        E, M = lat.sweep_record(5, 2)           # launches (no whole graph) or the cluster path
        E2, M2 = lat.sweep_record(34, 17)       # a replayed graph of the launch path
        spins = lat.get_spins()
    with oracle.sweep_rounds(rounds):
        s = oracle.init_hot(L, seed)
        Eo, Mo = oracle.run(s, seed, 0.43, 0, 5, 2)
        Eo2, Mo2 = oracle.run(s, seed, 0.43, 5, 34, 17)
    np.testing.assert_array_equal(np.concatenate([E, E2]), np.concatenate([Eo, Eo2]))
    np.testing.assert_array_equal(np.concatenate([M, M2]), np.concatenate([Mo, Mo2]))
    np.testing.assert_array_equal(spins, s)
