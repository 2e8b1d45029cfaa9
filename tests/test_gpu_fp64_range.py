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


@pytest.mark.parametrize("rho", [2.0, 40.0])
def test_forces_away_from_rho0_do_not_go_one_by_one(L, pack, rho):
    """A pack at 2 and at 40 rho0, 504 and 549 us per step against 164 at rho0;
    1214 and 4120 when each large term of the force was an atomic of its own."""
    t1, t2 = (_step_time(L, pack, 1.0, r, bc=2) for r in (1.0, rho))
    assert t2 <= 5.0 * t1


@pytest.mark.parametrize("stencil", [G.D2Q9, G.D3Q19])
@pytest.mark.parametrize("fused", [0, 1])
@pytest.mark.parametrize("scale", [1.0, 1.3, 2.0, 40.0, 1e6])
def test_forces_at_any_density(L, stencil, fused, scale):
    """Forces of a flow, a density `scale` times rho0 (the link sums run in grid
    steps, one by one beyond their range, and both ways within one warp where the
    density varies across its edge): against the sum over links of the populations themselves.
    A sum of n terms of size t = max |f+ + f'| in any order: n^2 eps t."""
    if stencil == G.D2Q9:
        geo = G.build(0, (45, 33, 1), (1, 1, 1), [G.ball((20.37, 15.61, 0), 6.3)])
    else:
        geo = G.build(1, (19, 18, 17), (1, 1, 1), [G.ball((9.3, 8.6, 8.1), 4.7)])
    rng = np.random.default_rng(2)
    e = G.velocity_set(stencil)
    with L.Lattice(geo, precision=L.LBM_FP64, tau=0.8, bc=0) as lat:
        lat.set_tuning(bulk_shape=1, fused=fused)
        u = np.zeros((geo.N, 3))
        u[:, 0] = 0.02
        u[geo.solid != 0] = 0
        lat.init_equilibrium(scale * rng.uniform(0.9, 1.1, geo.N), u)
        f = lat.distributions()
        lat.step(1)
        F = lat.forces(1)[0]
    # half-way links at rest hand f+_i' back: each exchanges 2 f+_i' e_i'
    lk = geo.links
    t = 2.0 * f[lk["dir"], lk["node"]]
    ref = (t[:, None] * e[lk["dir"]]).sum(0)
    n = len(lk)
    assert np.all(np.abs(F - ref) <= n * n * np.finfo(float).eps * t.max()) and np.abs(ref[0]) > 0
