"""Spins to words: rows at every alignment of the input (16-byte rows, rows that
begin at offset 0 and 2 of a 4-byte word, an input at an odd address), last
words of one spin and of 21, any positive value up and any other down; and a
series of states whose device counter is read back by a captured graph's path."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ising():
    import paper_1811_04384_gb300 as p
    p.load()
    return p


@pytest.mark.parametrize("L", [4, 6, 16, 42, 44, 62, 64, 66, 126, 130, 336, 338, 1040, 1042, 4100])
@pytest.mark.parametrize("offset", [0, 1, 2, 4])
@pytest.mark.parametrize("pinned", [False, True])
def test_alignments(ising, L, offset, pinned):
    import torch
    values = np.array([1, 127, 2, 64, -1, 0, -128, -127], dtype=np.int8)
    s = values[np.random.default_rng(L + offset).integers(0, 8, size=(L, L))]
    buf = torch.empty(L * L + 16, dtype=torch.int8, pin_memory=pinned).numpy()
    view = buf[offset:offset + L * L].reshape(L, L)
    view[:] = s
    with ising.Lattice(L, 1) as lat:
        lat.set_spins(view)
        spins, words = lat.get_spins(), lat.get_words()
        with ising.Lattice(L, 1) as other:
            other.set_words(words)
            np.testing.assert_array_equal(other.get_spins(), spins)
    np.testing.assert_array_equal(spins, np.where(s > 0, 1, -1))


@pytest.mark.parametrize("L", [3100, 3104])
def test_states_then_other_paths(ising, L):
    """Launch-path states, then sweeps that count from the device's counter."""
    rng = np.random.default_rng(7)
    states = [np.where(rng.random((L, L)) < 0.5, 1, -1).astype(np.int8) for _ in range(3)]
    with ising.Lattice(L, 9) as a, ising.Lattice(L, 9) as b:
        for lat in (a, b):
            lat.set_beta(0.43)
        E, M = a.run_states(states, 4, 2)
        for k, s in enumerate(states):
            b.set_spins(s)
            Eb, Mb = b.sweep_record(4, 2)
            np.testing.assert_array_equal(E[k], Eb)
            np.testing.assert_array_equal(M[k], Mb)
        assert a.t == b.t == 12
        Ea, Ma = a.sweep_record(3, 1)
        Eb, Mb = b.sweep_record(3, 1)
        np.testing.assert_array_equal(Ea, Eb)
        np.testing.assert_array_equal(a.get_spins(), b.get_spins())
