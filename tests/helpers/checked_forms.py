"""The forms of the kernels that the small-lattice battery does not reach, run
against the checked build of the library (ISING_LIBRARY pointing at
libising_checked.so): each result compared with the oracle, then the device's
out-of-range record read back.  Prints one JSON line; exits non-zero on a
mismatch."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

import oracle  # noqa: E402
import paper_1811_04384_gb300 as p  # noqa: E402

BETA = 1.0 / 2.269
CASES = []


def case(name, got, want):
    _, violation = p.check_status()
    same = all(np.array_equal(np.asarray(g), np.asarray(w)) for g, w in zip(got, want))
    if violation or not same:
        print(json.dumps({"ok": False, "case": name, "violation": violation}))
        sys.exit(1)
    CASES.append(name)


def sweeps(name, L, n, every, path=None, clusters=0, layout=0):
    seed = 11 + L
    with p.Lattice(L, seed, layout=layout) as lat:
        if path is not None:
            lat.set_path(path)
        lat.set_clusters(clusters)
        lat.init_hot()
        lat.set_beta(BETA)
        E, M = lat.sweep_record(n, every)
        S = lat.get_spins()
    s = oracle.init_hot(L, seed)
    Eo, Mo = oracle.run(s, seed, BETA, 0, n, every)
    case(f"{name} L={L}", (E, M, S), (Eo, Mo, s))


def words(L, nstrips, n):
    seed = 5 + nstrips
    with p.Lattice(L, seed, layout=p.ISING_LAYOUT_COLUMN_INTERLEAVED) as lat:
        lat.init_hot()
        lat.set_chain(p.ISING_CHAIN_RANDOM_WORDS, nstrips)
        lat.set_beta(BETA)
        E, M = lat.sweep_record(n, 1)
        S = lat.get_spins()
    s = oracle.init_hot(L, seed)
    Eo, Mo = oracle.rw_run(s, seed, BETA, 0, n, nstrips)
    case(f"random words L={L} strips={nstrips}", (E, M, S), (Eo, Mo, s))


def pack(L, offset):
    rng = np.random.default_rng(L + offset)
    buf = np.empty(L * L + 16, dtype=np.int8)
    view = buf[offset:offset + L * L].reshape(L, L)
    view[:] = np.where(rng.random((L, L)) < 0.5, 1, -1)
    with p.Lattice(L, 1) as lat:
        lat.set_spins(view)
        S = lat.get_spins()
    case(f"spins in, L={L} offset={offset}", (S,), (view,))


def main():
    checked, _ = p.check_status()
    C, LAUNCHES, CI = p.ISING_PATH_CLUSTER, p.ISING_PATH_LAUNCHES, p.ISING_LAYOUT_COLUMN_INTERLEAVED
    for L in (4, 6, 64, 66, 70, 126, 128):                       # one warp: one and two words, a last lane of two rows
        sweeps("warp", L, 9, 2, path=p.ISING_PATH_RESIDENT)
    for L in (130, 258, 514, 896):                               # rows of 3 to 14 words, more than one phase, pieces
        sweeps("band", L, 33, 4, path=C, clusters=1)
    sweeps("band pieces", 296, 210, 7, path=C, clusters=1)
    for L in (34, 128, 898, 1008, 1026):                         # one cluster, one and two words a unit
        sweeps("cluster", L, 21, 3, path=C, clusters=1)
    sweeps("cluster, two units a thread", 1600, 3, 1, path=C, clusters=1)
    for L, G in ((330, 2), (1008, 3), (2016, 3)):
        sweeps(f"{G} clusters", L, 21, 3, path=C, clusters=G)
    for L, G in ((84, 1), (168, 1), (504, 1), (1008, 1), (1008, 2)):
        sweeps(f"interleaved, {G} clusters", L, 21, 3, path=C, clusters=G, layout=CI)
    for L in (84, 252, 1512, 1596):                              # split over the block's warps, and whole
        sweeps("interleaved launches", L, 5, 1, path=LAUNCHES, layout=CI)
    for L in (2340, 2342):                                       # several strips, in graphs and outside
        sweeps("launches", L, 3, 1, path=LAUNCHES)
    for L, strips in ((84, 42), (84, 1), (252, 84), (1008, 72), (1008, 21), (1008, 18)):
        words(L, strips, 2)
    for L, offset in ((64, 0), (66, 0), (66, 1), (130, 2), (1042, 4)):
        pack(L, offset)
    checked_after, violation = p.check_status()
    print(json.dumps({"ok": violation == 0, "checked": checked and checked_after, "violation": violation,
                      "cases": len(CASES)}))
    sys.exit(0 if violation == 0 else 2)


if __name__ == "__main__":
    main()
