"""FP64 lattices whose density is far from 1 or from rho0: the integer grid
follows rho0, and what is outside it goes back to doubles at no more than the
doubles' cost.  Times are the best of five runs of one program on the same
lattice; the bounds leave half of what each fault cost."""
import time

import numpy as np
import pytest

from paper_1903_01111_gb300 import geometry as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1903_01111_gb300 import lbm

    return lbm


def _step_time(L, geo, rho0, rho, tuning=None, steps=20, **kw):
    with L.Lattice(geo, precision=L.LBM_FP64, rho0=rho0, tau=0.8, **kw) as lat:
        if tuning:
            lat.set_tuning(**tuning)
        lat.init_equilibrium(np.full(geo.N, float(rho)))
        best = np.inf
        for _ in range(5):
            lat.synchronize()
            t = time.perf_counter()
            lat.step(steps)
            lat.synchronize()
            best = min(best, (time.perf_counter() - t) / steps)
        lat.check()
    return best


@pytest.fixture(scope="module")
def pack():
    return G.sphere_pack(128)


@pytest.mark.parametrize("rho0", [0.4, 1000.0])
def test_speed_does_not_depend_on_rho0(L, pack, rho0):
    """Ghost slots of the fused step: 431 against 211 us per step when their rest
    state was outside the grid of any rho0 but 1."""
    t1, t2 = (_step_time(L, pack, r, r, dict(bulk_shape=1, fused=1), bc=2) for r in (1.0, rho0))
    assert t2 <= 1.5 * t1
