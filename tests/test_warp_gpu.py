"""The on-chip path of small lattices (one warp, one bit per spin): lanes with
and without rows, a last lane of two rows, last words of 1 and 32 live bits,
thresholds of 2^32 and 0, several mask pieces; against the oracle bit for bit."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ising():
    import paper_1811_04384_gb300 as p
    p.load()
    return p


def check(ising, L, beta, n, every, start, rounds=10):
    seed = 0x0123456700000000 + L
    with ising.Lattice(L, seed) as lat, oracle.sweep_rounds(rounds):
        lat.set_path(ising.ISING_PATH_RESIDENT)
        if rounds == 7:
            lat.set_rng(ising.ISING_RNG_PHILOX4X32_7)
        lat.init_hot()
        lat.set_beta(beta)
        lat.t = start
        lat.sweep(3)
        E, M = lat.sweep_record(n, every)
        lat.sweep(1)
        t, spins = lat.t, lat.get_spins()
        s = oracle.init_hot(L, seed)
        oracle.run(s, seed, beta, start, 3, 3)
        Eo, Mo = oracle.run(s, seed, beta, start + 3, n, every)
        oracle.run(s, seed, beta, start + 3 + n, 1, 1)
    np.testing.assert_array_equal(E, Eo)
    np.testing.assert_array_equal(M, Mo)
    np.testing.assert_array_equal(spins, s)
    assert t == start + 4 + n


@pytest.mark.parametrize("L", [4, 6, 42, 62, 64, 66, 68, 70, 84, 86, 126, 128])
@pytest.mark.parametrize("beta,every", [(0.0, 1), (1 / 2.269, 3), (4.0, 5)])
def test_against_oracle(ising, L, beta, every):
    check(ising, L, beta, 23, every, 2**32 - 9)


@pytest.mark.parametrize("L,every,rounds", [(128, 4500, 10), (126, 1, 7)])
def test_pieces(ising, L, every, rounds):
    check(ising, L, 0.44, 9001 if rounds == 10 else 50, every, 0, rounds)


# sweeps past the layers of one draw launch: equal to the fused launches
def test_layers(ising):
    out = []
    for path in (ising.ISING_PATH_RESIDENT, ising.ISING_PATH_LAUNCHES):
        with ising.Lattice(4, 5) as lat:
            lat.set_path(path)
            lat.init_hot()
            lat.set_beta(0.4)
            E, M = lat.sweep_record(65535 + 70, 65535 // 5)
            out.append((E, M, lat.get_spins()))
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
