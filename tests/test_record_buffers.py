"""The record arrays that the binding hands to the library, on the CPU: E's and
M's entries for counts of every integer type, whose own range the sizes and byte
offsets may pass."""
import ctypes
import types

import numpy as np
import pytest

import paper_1811_04384_gb300 as p


def fake_record(seen):
    @ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p, ctypes.c_int64, ctypes.c_int64, ctypes.c_void_p, ctypes.c_void_p)
    def ising_sweep_record(h, n, every, E, M):
        seen.append((n // every, M - E))
        if M - E == 8 * (n // every):          # both series fit one buffer: E's end is M's start
            for k in range(n // every):
                ctypes.c_int64.from_address(E + 8 * k).value = k
                ctypes.c_int64.from_address(M + 8 * k).value = -k
        return 0
    return ising_sweep_record


@pytest.mark.parametrize("n", [np.int8(100), np.uint8(200), np.int16(5000), np.int16(20000), np.uint16(40000),
                               np.int32(300), np.int64(300), 300])
def test_counts_of_any_integer_type(monkeypatch, n):
    seen = []
    record = fake_record(seen)
    monkeypatch.setattr(p, "load", lambda: types.SimpleNamespace(ising_sweep_record=record))
    lat = object.__new__(p.Lattice)
    lat._h = None
    E, M = lat.sweep_record(n, 1)
    assert seen == [(int(n), 8 * int(n))]
    np.testing.assert_array_equal(E, np.arange(int(n)))
    np.testing.assert_array_equal(M, -np.arange(int(n)))


@pytest.mark.parametrize("n", [10.0, "10"])
def test_counts_that_are_no_integers(monkeypatch, n):
    monkeypatch.setattr(p, "load", lambda: types.SimpleNamespace(ising_sweep_record=fake_record([])))
    lat = object.__new__(p.Lattice)
    lat._h = None
    with pytest.raises(TypeError):
        lat.sweep_record(n, 1)


@pytest.mark.parametrize("counts", [[], [0], [3], [2, 0, 5], [1] * 32, list(range(33)), [4] * 300])
def test_arrays_of_a_batch(counts):
    arrays, addresses = p._records(counts)
    assert len(arrays) == len(addresses) == len(counts)
    for k, (a, n) in enumerate(zip(arrays, counts)):
        assert a.shape == (n,) and a.dtype == np.int64 and a.flags["C_CONTIGUOUS"] and not a.any()
        if n:
            assert addresses[k] == a.ctypes.data
        a[:] = k
    for k, a in enumerate(arrays):
        assert (a == k).all()                         # none lies over another


@pytest.mark.parametrize("counts,error", [([1, -1], ValueError), ([2.0], TypeError)])
def test_arrays_of_a_batch_refused(counts, error):
    with pytest.raises(error):
        p._records(counts)


def test_arrays_of_one_replica_take_microseconds():
    """Two such calls are in every Batch.sweep (20 us each while they used NumPy
    throughout, against the 6 us of an array and a ctypes pointer)."""
    import timeit

    def pointer():
        a = np.zeros(20, dtype=np.int64)
        return a, p._ptr_array([a], ctypes.c_int64)
    def once():
        a, b = (min(timeit.repeat(f, number=200, repeat=20)) for f in (lambda: p._records([20]), pointer))
        return a / b
    assert min(once() for _ in range(3)) < 2
