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


# ------------------------------------------------------------- link values --

QS = (1e-300, 1e-6, 1e-3, 0.1, 0.3, 0.4999999, 0.5, 0.5000001, 0.7, 0.999, 1.0)


def _links_case(stencil, kind, seed):
    """A lattice with solid nodes all over, VIBB links of every q, three bodies
    (and none) in turn, walls that move; populations of `kind` (test_gpu_fixed64)
    for rho0 = 1."""
    from test_gpu_fixed64 import _masked, _state

    rng = np.random.default_rng([seed, stencil])
    shape = (37, 23, 1) if stencil == G.D2Q9 else (13, 9, 8)
    N = int(np.prod(shape))
    geo = _masked(stencil, shape, (rng.random(N) < 0.07).astype(np.uint8), bc=-1)
    lk = geo.links
    lk["q"] = rng.choice(QS, len(lk))
    lk["body"] = rng.integers(-1, 3, len(lk))
    lk["uw"] = rng.uniform(-1, 1, (len(lk), 3)) * (0.7 if kind == "fast" else 0.05)
    if stencil == G.D2Q9:
        lk["uw"][:, 2] = 0
    return geo, _state(stencil, N, 1.0, kind, rng) * (geo.solid == 0)


def _second_nodes(geo):
    """x_ff of every link (x_f where that is solid)."""
    n = geo.links["node"]
    e = G.velocity_set(geo.stencil)[geo.links["dir"]].astype(int)
    x = np.stack(np.unravel_index(n, (geo.nz, geo.ny, geo.nx)))[::-1]
    y = (x - e.T) % np.array([[geo.nx], [geo.ny], [geo.nz]])
    ff = y[0] + geo.nx * (y[1] + geo.ny * y[2])
    return np.where(geo.solid[ff] != 0, n, ff)


def _link_magnitudes(geo, f, rho0, local_rho):
    """Per link: the sum of the magnitudes of the terms of its value, with the
    change that one eps of each moment's terms makes in it, and the square of how
    much the moments of its two nodes cancel."""
    from test_gpu_fixed64 import _weights

    e, w = _weights(geo.stencil)
    lk = geo.links
    n, d, q = lk["node"], lk["dir"], lk["q"]
    ff = _second_nodes(geo)
    rho, a = f.sum(0), np.abs(f).sum(0)
    with np.errstate(all="ignore"):
        u = np.abs(e.T @ f / rho)
        cond = a / np.abs(rho)
        amp = cond ** 2
    p, m = 2 * q, np.abs(1 - 2 * q)

    def K(v, c):  # 1 + 3 e.u + 4.5 (e.u)^2 - 1.5 u.u and its change with an error c eps of u
        s = v.sum(0)
        return 1 + 3 * s + 6 * s ** 2 + (3 + 12 * s) * c

    rd = np.where(local_rho & (q > 0.5), np.abs(rho[n]), p * np.abs(rho[n]) + m * np.abs(rho[ff]))
    with np.errstate(all="ignore"):
        ud = u[:, n] + u[:, ff] + np.abs(lk["uw"].T)
        M = w[d] * rd * K(ud, cond[n] + cond[ff]) + 6 * w[d] * rho0 * np.abs(lk["uw"]).sum(1)
        for k, c in ((n, p), (ff, m)):
            M = M + c * rd / np.abs(rho[k]) * (np.abs(f[d, k]) + w[d] * np.abs(rho[k]) * K(u[:, k], cond[k]))
    return M, np.maximum(1.0, np.maximum(amp[n], amp[ff]))


@pytest.mark.parametrize("kind", ["plain", "fast", "density", "odd"])
@pytest.mark.parametrize("rho0", [1.0, 0.75, 1.4999, 3e-9, 1.7e12])
@pytest.mark.parametrize("local_rho", [0, 1])
@pytest.mark.parametrize("stencil", [G.D2Q9, G.D3Q19])
def test_fp64_links_in_and_out_of_the_grid(L, stencil, local_rho, rho0, kind):
    """One step from given populations, in both step forms, against the oracle.
    A link value rounds about forty operations on terms of total size M, its
    moments carry the rounding of their populations amplified by `amp`, and a
    collision's outputs are at most 4 times its inputs' errors plus 64 eps of
    their sum: 256 eps (sum |f| + sum M amp) of the node.  A force sums its
    links: 64 eps M amp each and n eps of the sum of the terms."""
    import oracle as O

    geo, f0 = _links_case(stencil, kind, 11)
    f0 = f0 * rho0
    eps = np.finfo(float).eps
    cfg = O.make_config(stencil=stencil, nx=geo.nx, ny=geo.ny, nz=geo.nz, tau=0.8, rho0=rho0, bc=2, vibb_density=local_rho)
    st = O.State(f0.copy(), *O.moments(cfg, geo.solid, f0))
    Fr = O.run(cfg, geo.solid, geo.links, st, 1, nbody=3)
    fl = geo.solid == 0
    M, amp = _link_magnitudes(geo, f0, rho0, local_rho)
    from test_gpu_fixed64 import _pull, _weights

    e, w = _weights(stencil)
    lk = geo.links
    pulled = _pull(stencil, f0, (geo.nx, geo.ny, geo.nz))  # (from solid nodes: zeros)
    S, net = np.abs(pulled).sum(0), pulled.sum(0)
    np.add.at(S, lk["node"], M * amp)
    # the collision divides by the density, which the links may nearly cancel
    rho1 = np.abs(st.rho)
    with np.errstate(all="ignore"):
        S = S * np.maximum(1.0, (S / rho1) ** 2)
    t = np.abs(f0[lk["dir"], lk["node"]]) + M + 2 * w[lk["dir"]] * rho0
    for fused in (0, 1):
        with L.Lattice(geo, precision=L.LBM_FP64, tau=0.8, rho0=rho0, bc=2, vibb_density=local_rho) as lat:
            lat.set_tuning(bulk_shape=1, fused=fused)
            lat.init_equilibrium()
            lat.set_distributions(f0)
            lat.step(1)
            f, F = lat.distributions(), lat.forces(3)
        assert np.all(np.abs(f - st.fp)[:, fl] <= 256 * eps * S[fl]), (fused, np.nanmax((np.abs(f - st.fp) / S)[:, fl]))
        for b in range(3):
            k = lk["body"] == b
            tol = eps * (64 * (M * amp)[k].sum() + k.sum() * t[k].sum())
            assert np.all(np.abs(F[b] - Fr[b]) <= tol), (fused, b)


@pytest.mark.parametrize("fused", [0, 1])
@pytest.mark.parametrize("stencil", [G.D2Q9, G.D3Q19])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_fp64_links_keep_non_finite_values_visible(L, stencil, fused, bad):
    """One such population reaches the node it streams to and, through the
    moments of its node, every link that reads them, and no other node or body."""
    geo, f0 = _links_case(stencil, "plain", 12)
    lk = geo.links
    ff = _second_nodes(geo)
    n = int(lk["node"][len(lk) // 2])
    f0[5, n] = bad
    with L.Lattice(geo, precision=L.LBM_FP64, tau=0.8, bc=2) as lat:
        lat.set_tuning(bulk_shape=1, fused=fused)
        lat.init_equilibrium()
        lat.set_distributions(f0)
        lat.step(1)
        f, F = lat.distributions(), lat.forces(3)
        with pytest.raises(L.LBMError):
            lat.check()
    e = G.velocity_set(stencil)
    x = np.array(np.unravel_index(n, (geo.nz, geo.ny, geo.nx)))[::-1]
    to = (x + e[5].astype(int)) % (geo.nx, geo.ny, geo.nz)
    reads = (lk["node"] == n) | (ff == n)
    expect = np.zeros(geo.N, bool)
    expect[to[0] + geo.nx * (to[1] + geo.ny * to[2])] = True
    expect &= geo.solid == 0
    expect[lk["node"][reads]] = True
    assert np.array_equal(~np.isfinite(f).all(0), expect)
    assert [not np.isfinite(F[b]).all() for b in range(3)] == [bool((reads & (lk["body"] == b)).any()) for b in range(3)]


# ----------------------------------------------------------------- memory --

def test_fused_link_weights_are_held_only_for_the_fused_step(L):
    """Bodies in turn make the fused step's link order another than the link
    kernel's, and its velocity weights (24 B a link) a second copy: not held by
    the split step that FP64 D3Q19 starts with, and the same step either way."""
    geo, f0 = _links_case(G.D3Q19, "plain", 13)
    with L.Lattice(geo, precision=L.LBM_FP64, tau=0.8, bc=2) as lat:
        lat.init_equilibrium()
        held = lat.info().device_bytes
        out = []
        for fused in (0, 1, 0, 1):
            lat.set_tuning(bulk_shape=1, fused=fused)
            assert lat.info().device_bytes == held + fused * 24 * len(geo.links)
            lat.set_distributions(f0)
            lat.step(2)
            out.append(lat.distributions())
    assert np.array_equal(out[0], out[2]) and np.array_equal(out[1], out[3])
    assert np.abs(out[0] - out[1]).max() <= 1e-14
    # chosen before the geometry
    with L.Lattice(None, stencil=1, nx=geo.nx, ny=geo.ny, nz=geo.nz, precision=L.LBM_FP64, tau=0.8, bc=2) as lat:
        lat.set_tuning(bulk_shape=1, fused=1)
        lat.set_geometry(geo.solid, geo.links)
        lat.init_equilibrium()
        lat.set_distributions(f0)
        lat.step(2)
        assert np.array_equal(lat.distributions(), out[1])


def test_force_slots_of_a_monitored_loop_are_counted(L):
    geo = G.build(0, (45, 33, 1), (1, 1, 1), [G.ball((20.37, 15.61, 0), 6.3)])
    with L.Lattice(geo, precision=L.LBM_FP64, tau=0.8, bc=2) as lat:
        lat.init_equilibrium()
        held = lat.info().device_bytes
        lat.step_forces(100, 0)
        assert lat.info().device_bytes == held + 100 * 3 * 8 * lat.info().n_bodies


# ----------------------------------------------------------------- batches --

def test_domains_with_strong_forces_equal_themselves_alone(L):
    """A domain's force beyond the grid's (|g| > rho0 / 512) sends its collisions
    to doubles, not its links: the same bits alone and in a batch whose other
    domain has a weak force."""
    from test_gpu_fixed64 import _masked

    rng = np.random.default_rng(4)
    nx, n, forces = 33, 20, [(0.01, 0.0, 0.0), (1e-4, 0.0, 0.0)]
    parts = []
    for _ in forces:
        solid = (rng.random((n, nx)) < 0.05).astype(np.uint8)
        solid[0] = solid[-1] = 1
        parts.append(_masked(G.D2Q9, (nx, n, 1), solid.reshape(-1), q=0.3, bc=-1))
    both = _masked(G.D2Q9, (nx, 2 * n, 1), np.concatenate([p.solid for p in parts]), q=0.3, bc=-1)
    kw = dict(precision=L.LBM_FP64, bc=2, vibb_density=1)
    with L.Lattice(both, domains=[dict(lo=n * k, n=n, nx=nx, tau=0.9, g=g) for k, g in enumerate(forces)], tau=0.9,
                   **kw) as lat:
        lat.init_equilibrium()
        lat.step(7)
        f = lat.distributions().reshape(9, 2, -1)
    for k, g in enumerate(forces):
        with L.Lattice(parts[k], tau=0.9, g=g, **kw) as lat:
            lat.init_equilibrium()
            lat.step(7)
            assert np.array_equal(f[:, k], lat.distributions()), k
