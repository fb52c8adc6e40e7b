"""Learned moves where the network's value leaves FP32's range."""
import numpy as np
import pytest

from tests.test_gpu_parity import hq  # noqa: F401
from workloads import HolsteinParams, random_fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,block", [(4, 4, False), (8, 4, True), (4, 4, True)])
def test_moves_into_an_infinite_barrier_are_rejected(hq, nx, ny, block):  # noqa: F811
    """f = 0 below z = 1 at the patch's centre and -2^140 (z - 1), minus infinity in FP32, above: no move of a chain
    that starts below the barrier passes it, and nothing else of the chain is touched by the rejected values."""
    p = HolsteinParams(nx=nx, ny=ny, beta=0.8, seed=99)
    X0 = random_fields(p, 3, seed=5, scale=0.0, offset=-p.g)  # z = X + g = 0
    th = np.zeros(hq.HQ_NN_PARAMS)
    th[10 * 64] = 2.0 ** 60              # input 10: the patch's own site and slice
    th[25 * 64] = -(2.0 ** 60)           # hidden unit 0 of layer 1: 2^60 (z - 1)
    th[26 * 64] = 2.0 ** 60              # of layer 2: 2^120 (z - 1)
    th[26 * 64 + 64 * 64 + 64] = -(2.0 ** 20)
    eng = hq.Engine(p, 3)
    eng.attach_network(1, 1)
    eng.set_params(th)
    eng.set_fields(X0)
    for _ in range(6):
        eng.cumulative(1, 1, global_=block)
    z = eng.get_fields() + p.g
    st = eng.learned_stats()
    obs = eng.observables()
    for c in range(3):
        assert obs[c]["status"] == 0
        assert 0 < st[c]["inner_local_accepted"] < st[c]["inner_local_proposed"]
        assert z[c].max() < 1.0 + 1e-4
        assert np.isfinite(st[c]["last_pc"])
    assert any(s["cumulative_accepted"] for s in st)
    eng.close()
