"""D2Q9 step kernels at their edges: pairs of neighbouring nodes against one
node per thread (FP32 BGK: the same bits), groups with links taken by a warp or
by a whole block, and open columns written by their neighbours' threads."""
import time

import numpy as np
import pytest

from paper_1903_01111_gb300 import batch as B
from paper_1903_01111_gb300 import geometry as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1903_01111_gb300 import lbm

    return lbm


def _start(geo, seed):
    rng = np.random.default_rng(seed)
    u = np.zeros((geo.N, 3))
    u[:, :2] = rng.uniform(-0.03, 0.03, (geo.N, 2))
    u[geo.solid != 0] = 0
    return 1.0 + rng.uniform(-0.01, 0.01, geo.N), u


def _run(L, geo, steps, domains=None, tuning=None, **kw):
    lat = L.Lattice(geo, domains=domains, **kw)
    if tuning:
        lat.set_tuning(**tuning)
    lat.init_equilibrium(*_start(geo, 3))
    lat.step(steps)
    out = lat.distributions(), lat.forces()
    lat.close()
    return out


def _geometries():
    yield "box 1x1", G.build(0, (1, 1, 1), (1, 1, 1), []), None, {}
    yield "box 2x3", G.build(0, (2, 3, 1), (1, 1, 1), []), None, {}
    yield "box 31x5", G.build(0, (31, 5, 1), (1, 1, 1), []), None, {}
    yield "box 33x64", G.build(0, (33, 64, 1), (1, 1, 1), []), None, {}
    yield "rotor 45x33", G.build(0, (45, 33, 1), (1, 1, 1), [G.ball((20.37, 15.61, 0), 6.3, omega=(0, 0, 0.004))]), None, {}
    geo = G.cylinder_channel(nx=121, ny_fluid=30, center=(30.37, 15.61), radius=4.3)
    yield "channel", geo, None, dict(inlet_umax=0.05, inlet_y0=0.5, inlet_y1=30.5)
    b = B.stack(B.draw_channels(3, seed=2, nx_range=(40, 61), ny_range=(24, 31), r_range=(3.0, 4.0), n_cyl=(1, 2)))
    yield "batch", b.geometry, b.domains, dict(inlet_y0=0.0, inlet_y1=1.0)


CASES = list(_geometries())


@pytest.mark.parametrize("g", [(0.0, 0.0, 0.0), (2e-5, -1e-5, 0.0)])
@pytest.mark.parametrize("case", range(len(CASES)), ids=[c[0] for c in CASES])
def test_pairs_have_the_bits_of_single_nodes(L, case, g):
    _, geo, domains, kw = CASES[case]
    if domains is not None:
        domains = [dict(d, g=g) for d in domains]
    ref = None
    for shape in (1, 0, 2, 3, 4, 5, 6, 7):
        f, F = _run(L, geo, 7, domains, dict(bulk_shape=shape, fused=0), precision=L.LBM_FP32_SHIFTED, tau=0.7, g=g, **kw)
        if ref is None:
            ref = f
        assert np.array_equal(f, ref), shape


@pytest.mark.parametrize("collision", ["bgk", "mrt"])
@pytest.mark.parametrize("prec", ["fp64", "fp32s"])
@pytest.mark.parametrize("name", ["whole blocks", "warps", "warps, one body per wall"])
def test_linked_groups_by_warps_and_by_blocks(L, name, prec, collision):
    """The step with the links in the pull pass against the link kernel and the
    bulk pass: few groups with links (a block on each) and more than the chip
    holds blocks (a warp on each); FP64 differs in the order of a few roundings
    (20 steps, 1e-13), FP32 by 4 steps eps of the deviations, as in the parity
    tests."""
    if name == "whole blocks":
        geo = G.cylinder_channel(nx=200, ny_fluid=40, center=(50.37, 20.61), radius=6.3)
    else:
        two = name != "warps"
        geo = G.channel(0, 6007, 24, q_lo=0.3, q_hi=0.7, u_hi=(0.01, 0, 0), force_lo=0, force_hi=1 if two else 0)
    kw = dict(precision=L.LBM_FP64 if prec == "fp64" else L.LBM_FP32_SHIFTED, tau=0.7,
              collision=L.LBM_MRT if collision == "mrt" else L.LBM_BGK)
    if geo.open_x[0]:
        kw.update(inlet_umax=0.05, inlet_y0=0.5, inlet_y1=40.5)
    else:
        kw.update(g=(1e-5, 0, 0))
    steps = 20
    (fa, Fa), (fb, Fb) = (_run(L, geo, steps, None, dict(bulk_shape=1, fused=k), **kw) for k in (1, 0))
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None]
    fl = geo.solid == 0
    if prec == "fp64":
        tol = 1e-13
    else:
        tol = 4 * steps * float(np.finfo(np.float32).eps) * np.abs((fb - w)[:, fl]).max()
    assert np.abs(fa - fb).max() <= tol
    assert np.abs(Fa - Fb).max() <= max(np.abs(Fb).max(), 1e-3) * (1e-10 if prec == "fp64" else 1e-4) + len(geo.links) * tol
    # the monitored loop leaves the same state and the last force
    lat = L.Lattice(geo, **kw)
    lat.set_tuning(bulk_shape=1, fused=1)
    lat.init_equilibrium(*_start(geo, 3))
    series = lat.step_forces(steps, 0)
    assert np.array_equal(lat.distributions(), fa)
    np.testing.assert_allclose(series[-1], lat.force(0), rtol=0, atol=0)
    lat.close()


@pytest.mark.parametrize("g", [(0.0, 0.0, 0.0), (2e-5, -1e-5, 0.0)])
@pytest.mark.parametrize("case", [c for c in range(len(CASES)) if not CASES[c][0].startswith("box")],
                         ids=[c[0] for c in CASES if not c[0].startswith("box")])
def test_adjoint_pairs_against_one_node_in_doubles(L, case, g):
    """The FP32 D2Q9 adjoint (pairs; odd row lengths, seams, open columns,
    domains with rates of their own) against FP64's one node per thread, every
    link and every domain: 1e-3 of the largest entry, the bound of the FP32
    adjoint test at 300 steps."""
    _, geo, domains, kw = CASES[case]
    if domains is not None:
        domains = [dict(d, g=g) for d in domains]
    out = []
    for prec in (L.LBM_FP64, L.LBM_FP32_SHIFTED):
        with L.Lattice(geo, domains=domains, precision=prec, tau=0.7, g=g, **kw) as lat:
            lat.init_equilibrium(u=_smooth(geo))
            w = np.tile([1.0, 0.3, 0.0], (lat.info().n_bodies, 1))
            out.append(L.lbm_adjoint_step(lat.h, -1, w, 40, 9))
    (_, qa, ta, _), (_, qb, tb, _) = out
    assert np.abs(qa).max() > 0 and np.abs(qb - qa).max() <= 1e-3 * np.abs(qa).max()
    ta, tb = np.atleast_1d(ta), np.atleast_1d(tb)
    assert np.abs(ta).max() > 0 and np.abs(tb - ta).max() <= 1e-3 * np.abs(ta).max()


def _smooth(geo):
    x = np.arange(geo.N) % geo.nx
    y = np.arange(geo.N) // geo.nx
    u = np.zeros((geo.N, 3))
    u[:, 0] = 0.03 + 0.01 * np.sin(2 * np.pi * y / geo.ny)
    u[:, 1] = 0.01 * np.cos(2 * np.pi * x / geo.nx)
    u[geo.solid != 0] = 0
    return u


@pytest.mark.parametrize("prec", ["fp64", "fp32s"])
def test_inlet_needs_a_second_column(L, prec):
    """The inlet column is filled from the fluid node at x = 1; a lattice of one
    column has none, and the node after its last row would be beyond the storage
    (32 rows fill it exactly)."""
    lat = L.Lattice(None, stencil=0, nx=1, ny=32, nz=1, periodic=(0, 1, 1), tau=0.8, inlet=1, inlet_umax=0.05, inlet_y0=-0.5,
                    inlet_y1=31.5, precision=L.LBM_FP64 if prec == "fp64" else L.LBM_FP32_SHIFTED)
    with pytest.raises(L.LBMError) as ex:
        lat.set_geometry(np.zeros(32, np.uint8), np.zeros(0, G.LINK_DTYPE))
    assert ex.value.status == L.LBM_ERR_INVALID_ARG and "inlet" in str(ex.value)
    lat.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32s"])
def test_states_beyond_l2_in_every_form(L, prec):
    """More state than L2 keeps (rows end in partial groups, and the kernels
    prefetch ahead, past the end of the storage in its last blocks): one node and
    two per thread against the sequential walk, which does not prefetch, on a box
    (FP32: the same bits), and both step forms with bodies."""
    precision = L.LBM_FP64 if prec == "fp64" else L.LBM_FP32_SHIFTED
    shape = (1501, 1003, 1)
    box = G.build(0, shape, (1, 1, 1), [])
    ref = _run(L, box, 3, None, dict(bulk_shape=6, fused=0), precision=precision, tau=0.7)[0]
    for s in (1, 4, 2):
        f = _run(L, box, 3, None, dict(bulk_shape=s, fused=0), precision=precision, tau=0.7)[0]
        assert np.array_equal(f, ref) if prec == "fp32s" else np.abs(f - ref).max() <= 1e-14, s
    geo = G.build(0, shape, (1, 1, 1), [G.ball((x, y, 0), 9.3) for x in (40.3, 900.7, 1480.2) for y in (30.1, 970.6)])
    fa, fb = (_run(L, geo, 3, None, dict(bulk_shape=4, fused=k), precision=precision, tau=0.7)[0] for k in (0, 1))
    h = np.abs(fa - np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None])[:, geo.solid == 0].max()
    assert np.abs(fa - fb).max() <= (1e-13 if prec == "fp64" else 4 * 3 * float(np.finfo(np.float32).eps) * h)


@pytest.mark.parametrize("prec", ["fp64", "fp32s"])
def test_small_lattices_do_not_crowd_themselves_out(L, prec):
    """A long run of steps of a lattice of some 200 blocks: kernels that start
    early must not crowd each other out (32^3 nodes took 4.5 us per step in FP32
    against 3.8 at 40^3, 28^3 7.5 in FP64 against 4.4 at 24^3; now 2.8 and 4.2, 4.2
    and 3.5)."""
    precision = L.LBM_FP64 if prec == "fp64" else L.LBM_FP32_SHIFTED

    def us(m):
        geo = G.build(1, (m, m, m), (1, 1, 1), [])
        with L.Lattice(geo, precision=precision, tau=0.8) as lat:
            lat.init_equilibrium()
            best = np.inf
            for _ in range(6):
                lat.synchronize()
                t = time.perf_counter()
                lat.step(300)
                lat.synchronize()
                best = min(best, (time.perf_counter() - t) / 300 * 1e6)
        return best

    if prec == "fp32s":
        assert us(32) <= 1.1 * us(40)
    else:
        assert us(28) <= 1.45 * us(24)


@pytest.mark.parametrize("prec", ["fp64", "fp32s"])
def test_graphs_of_a_small_lattice_are_its_steps(L, prec):
    """Runs of steps on a small lattice of untouched tuning (graphs of 16, 8 and 4)
    against steps launched one by one: the same bits and forces, from odd steps too, and
    when the caller captures them."""
    import torch

    precision = L.LBM_FP64 if prec == "fp64" else L.LBM_FP32_SHIFTED
    geo = G.cylinder_channel(nx=121, ny_fluid=30, center=(30.37, 15.61), radius=4.3)
    kw = dict(precision=precision, tau=0.7, inlet_umax=0.05, inlet_y0=0.5, inlet_y1=30.5)
    s = torch.cuda.Stream()
    with L.Lattice(geo, **kw) as a, L.Lattice(geo, **kw) as b, L.Lattice(geo, stream=s.cuda_stream, **kw) as c:
        t = b.tuning()
        b.set_tuning(bulk_shape=t.bulk_shape, link_threads=t.link_threads, link_seq=t.link_seq, fused=t.fused, graph_steps=2)
        for lat in (a, b, c):
            lat.init_equilibrium(*_start(geo, 3))
        for n in (1, 100, 33, 2, 31, 12, 5, 7, 16):
            a.step(n)
            b.step(n)
            c.step(n)
            assert np.array_equal(a.distributions(), b.distributions()), n
            scale = np.abs(b.forces()).max()
            assert np.abs(a.forces() - b.forces()).max() <= 1e-12 * scale + (0 if prec == "fp64" else 1e-5 * scale)
        assert a.info().step == b.info().step == 207
        a.step(1)
        b.step(1)
        c.step(1)
        c.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            c.step(40)
        with torch.cuda.stream(s):
            g.replay()
        c.synchronize()
        b.step(40)
        assert np.array_equal(c.distributions(), b.distributions())


def test_several_small_lattices_are_not_bound_by_launches(L):
    """Three 32 x 24 lattices stepped in turn by one host thread: 1.9 us per step
    when each step was a launch, 1.0 in graphs of 16; one lattice 2.6."""
    geo = G.channel(0, 32, 24, q_lo=0.3, q_hi=0.3)
    lats = [L.Lattice(geo, precision=L.LBM_FP32_SHIFTED, tau=0.8, bc=2, g=(1e-6, 0, 0)) for _ in range(3)]
    for lat in lats:
        lat.init_equilibrium()

    def us(which):
        best = np.inf
        for _ in range(6):
            for lat in lats:
                lat.synchronize()
            t = time.perf_counter()
            for k in range(30):
                which[k % len(which)].step(160)
            for lat in lats:
                lat.synchronize()
            best = min(best, (time.perf_counter() - t) / 30 / 160 * 1e6)
        return best

    one, three = us(lats[:1]), us(lats)
    for lat in lats:
        lat.close()
    assert three <= 0.55 * one
