"""Epochs of one, two and four lanes (the running jobs' sites set the number)
give each job its own lattice's results."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sides", [[64, 130], [2048] * 4 + [66], [2500, 2048, 3000, 64] * 2])
def test_lanes(sides):
    import paper_1811_04384_gb300 as ising
    from paper_1811_04384_gb300 import serving
    ising.load()
    with serving.Server(256 << 20) as server:
        requests = [serving.Request(L, 0.44 + 0.01 * k, 100 + k, 3 + k % 3) for k, L in enumerate(sides)]
        for r in requests:
            server.submit(r)
        for r in requests:
            server.wait(r.id)
    for k, (L, r) in enumerate(zip(sides, requests)):
        with ising.Lattice(L, 100 + k) as lat:
            lat.init_hot()
            lat.set_beta(0.44 + 0.01 * k)
            E, M = lat.sweep_record(3 + k % 3, 1)
        np.testing.assert_array_equal(r.E, E)
        np.testing.assert_array_equal(r.M, M)
