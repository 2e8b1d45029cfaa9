"""FP64 collision on the integer grid and the field read-out, against plain
numpy in doubles: nodes inside and outside the grid's range (negative, tiny,
large and non-finite populations, other densities, strong forces) and tile
edges of the read-out.

Tolerance of one collision: both sides round a few dozen operations of
quantities no larger than S = sum |f_i| + |g| of the node (times the relaxation
factors, at most 3 for the rates used), so |difference| <= 64 eps64 S.  The
read-out: rho is one sum, u one sum and one quotient, 64 eps relative to S and
S / rho, eps of the storage precision (float sums) for FP32.
"""
import numpy as np
import pytest

from paper_1903_01111_gb300 import geometry as G

pytestmark = pytest.mark.gpu

EPS = float(np.finfo(np.float64).eps)


@pytest.fixture(scope="module")
def L():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1903_01111_gb300 import lbm

    return lbm


def _weights(stencil):
    e = G.velocity_set(stencil)
    n = np.abs(e).sum(1)
    w = np.array([4 / 9, 1 / 9, 1 / 36]) if stencil == G.D2Q9 else np.array([1 / 3, 1 / 18, 1 / 36])
    return e.astype(np.float64), w[n]


M9 = np.array([[1] * 9, [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1], [0, 1, 0, -1, 0, 1, -1, -1, 1],
               [0, -2, 0, 2, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1], [0, 0, -2, 0, 2, 1, 1, -1, -1],
               [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]], float)


def _collide(stencil, f, tau, g, mrt=False):
    e, w = _weights(stencil)
    g = np.asarray(g, float)[:, None]
    rho = f.sum(0)
    u = (e.T @ f + 0.5 * g) / rho
    eu, eg = e @ u, e @ g
    n = f - w[:, None] * rho * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * (u * u).sum(0))
    src = w[:, None] * (3 * (eg - (u * g).sum(0)) + 9 * eu * eg)
    if mrt:
        s = np.array([0.3, 1.5, 1.5, 0.3, 1.2, 0.3, 1.2, 1 / tau, 1 / tau])[:, None]
        return f - (M9.T / (M9 * M9).sum(1)) @ (s * (M9 @ n) - (1 - 0.5 * s) * (M9 @ src))
    return f - n / tau + (1 - 0.5 / tau) * src


def _pull(stencil, f, shape):
    nx, ny, nz = shape
    e = G.velocity_set(stencil)
    return np.stack([np.roll(f[i].reshape(nz, ny, nx), tuple(e[i][::-1]), (0, 1, 2)).reshape(-1) for i in range(len(e))])


def _state(stencil, N, rho0, kind, rng):
    """Post-collision populations of N nodes in the neighbourhood of rho0 and
    beyond it."""
    e, w = _weights(stencil)
    u = rng.uniform(-0.1, 0.1, (3, N))
    if stencil == G.D2Q9:
        u[2] = 0
    rho = rho0 * rng.uniform(0.9, 1.1, N)
    if kind == "fast":           # |u| up to 0.6: across the range's edge in velocity
        u *= 6.0
    if kind == "density":        # across its edges in density
        rho = rho0 * 10.0 ** rng.uniform(-3, 3, N)
    eu = e @ u
    f = w[:, None] * rho * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * (u * u).sum(0)) * rng.uniform(0.9, 1.1, (len(w), N))
    if kind == "odd":            # negative, zero, tiny populations here and there
        i, n = rng.integers(0, len(w), N), np.arange(N)
        f[i, n] *= rng.choice([-1.0, 0.0, 1e-12, 1e-300, 30.0], N)
    return f


@pytest.mark.parametrize("kind", ["plain", "fast", "density", "odd"])
@pytest.mark.parametrize("tau,rho0,g", [(0.8, 1.0, (0.0, 0.0, 0.0)), (0.53, 1.0, (1e-4, -2e-5, 3e-5)),
                                        (1.0, 0.75, (1e-4, 0.0, 0.0)), (50.0, 1.4999, (0.0, 1e-3, 0.0)),
                                        (0.7, 3e-9, (1e-13, 0.0, 0.0)), (0.9, 1.7e12, (1e8, 1e7, 0.0)),
                                        (0.6, 1.0, (0.01, 0.0, 0.0))])
@pytest.mark.parametrize("form", ["bgk2", "mrt2", "bgk3"])
def test_fp64_collision_in_and_out_of_the_grid(L, form, tau, rho0, g, kind):
    """One step of a solid-free box from given populations.  (0.01 exceeds the
    force the grid takes; a density range of 10^+-3 and |u| up to 0.6 leave it
    at some nodes.)"""
    stencil, shape = (G.D3Q19, (11, 7, 5)) if form == "bgk3" else (G.D2Q9, (37, 11, 1))
    if stencil == G.D2Q9:
        g = (g[0], g[1], 0.0)
    rng = np.random.default_rng([hash_of(form), hash_of(kind)])
    geo = G.build(stencil, shape, (1, 1, 1), [])
    f0 = _state(stencil, geo.N, rho0, kind, rng)
    ref = _collide(stencil, _pull(stencil, f0, shape), tau, g, form == "mrt2")
    S = np.abs(_pull(stencil, f0, shape)).sum(0) + np.abs(g).sum()
    # u enters squared over rho: populations that nearly cancel in rho amplify
    pulled = _pull(stencil, f0, shape)
    S = S * np.maximum(1.0, (np.abs(pulled).sum(0) / np.abs(pulled.sum(0))) ** 2)
    for shape_id in ((0, 1, 2, 3, 4, 5, 6, 7) if stencil == G.D2Q9 else (0, 1, 2)):
        lat = L.Lattice(geo, precision=L.LBM_FP64, tau=tau, rho0=rho0, g=g, bc=2,
                        collision=L.LBM_MRT if form == "mrt2" else L.LBM_BGK)
        lat.set_tuning(bulk_shape=shape_id)
        lat.init_equilibrium()
        lat.set_distributions(f0)
        lat.step(1)
        f = lat.distributions()
        lat.close()
        assert np.all(np.abs(f - ref) <= 64 * EPS * S), (shape_id, np.max(np.abs(f - ref) / S))


def hash_of(s):
    return sum(ord(c) * 131 ** k for k, c in enumerate(s)) % (1 << 31)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf, 1e308])
@pytest.mark.parametrize("stencil", [G.D2Q9, G.D3Q19])
def test_fp64_non_finite_populations_stay_visible(L, stencil, bad):
    shape = (9, 8, 7 if stencil == G.D3Q19 else 1)
    geo = G.build(stencil, shape, (1, 1, 1), [])
    f0 = _state(stencil, geo.N, 1.0, "plain", np.random.default_rng(1))
    f0[3, 17] = bad
    lat = L.Lattice(geo, precision=L.LBM_FP64, tau=0.7)
    lat.init_equilibrium()
    lat.set_distributions(f0)
    with np.errstate(all="ignore"):
        ref = _collide(stencil, _pull(stencil, f0, shape), 0.7, (0, 0, 0))
    lat.step(1)
    f = lat.distributions()
    if np.isfinite(ref).all() and np.all(ref.sum(0) > 0):  # (1e308 is a large but finite density)
        lat.check()
    else:
        with pytest.raises(L.LBMError):
            lat.check()
    lat.close()
    assert np.array_equal(np.isfinite(f).all(0), np.isfinite(ref).all(0))
    ok = np.isfinite(ref).all(0)
    assert np.all(np.abs(f[:, ok] - ref[:, ok]) <= 64 * EPS * np.abs(ref[:, ok]).sum(0))


@pytest.mark.parametrize("prec", ["fp64", "fp32s"])
@pytest.mark.parametrize("shape", [(1, 1, 1), (127, 1, 1), (128, 1, 1), (129, 3, 1), (31, 33, 1), (64, 65, 1), (13, 11, 9),
                                   (40, 16, 8)])
@pytest.mark.parametrize("body", [False, True])
def test_field_read_out_at_tile_edges(L, shape, body, prec):
    """rho and u from the populations themselves, zero off the fluid, whatever
    the outputs held before."""
    import torch

    stencil = G.D3Q19 if shape[2] > 1 else G.D2Q9
    if body and min(shape[:2]) < 9:
        pytest.skip("no room for a body")
    r = min(s for s in shape if s > 1) / 2.0 - 1.5 if body else 0
    geo = G.build(stencil, shape, (1, 1, 1), [G.ball([s / 2.0 + 0.3 for s in shape], r)] if body else [])
    g = (2e-4, -1e-4, 5e-5 if stencil == G.D3Q19 else 0.0)
    rng = np.random.default_rng(5)
    e, w = _weights(stencil)
    f0 = _state(stencil, geo.N, 1.0, "odd" if prec == "fp64" else "plain", rng)
    f0[:, ::7] = w[:, None]  # at rest: zero sums in shifted storage
    lat = L.Lattice(geo, precision=L.LBM_FP64 if prec == "fp64" else L.LBM_FP32_SHIFTED, tau=0.7, g=g)
    lat.init_equilibrium()
    lat.set_distributions(f0)
    f = lat.distributions()
    D = 3 if stencil == G.D3Q19 else 2
    rho = torch.full((geo.N,), 7.0, dtype=torch.float64, device="cuda")
    u = torch.full((D, geo.N), 7.0, dtype=torch.float64, device="cuda")
    lat.moments(rho, u)
    lat.synchronize()
    rho, u = rho.cpu().numpy(), u.cpu().numpy()
    rho_h, u_h = lat.moments()
    lat.close()
    assert np.array_equal(rho, rho_h) and np.array_equal(u, u_h)
    fl = geo.solid == 0
    assert np.all(rho[~fl] == 0) and np.all(u[:, ~fl] == 0)
    eps = EPS if prec == "fp64" else float(np.finfo(np.float32).eps)
    h = f - (0 if prec == "fp64" else w[:, None])
    S = np.abs(h).sum(0) + np.abs(g).sum() + (0 if prec == "fp64" else EPS / eps)
    r = np.where(fl, f.sum(0), 1.0)
    ur = (e.T @ f - 0.5 * np.asarray(g)[:, None])[:D] / r
    assert np.all(np.abs(rho - r)[fl] <= 64 * eps * S[fl])
    amp = (1 + np.abs(ur).max(0)) / np.abs(r)
    assert np.all(np.abs(u - ur)[:, fl] <= 64 * eps * (S * amp)[fl])


def _masked(stencil, shape, solid, q=0.5, bc=0, body=-1):
    """A periodic lattice with a mask: a link wherever a direction of a fluid
    node points into the solid, all of one rule."""
    nx, ny, nz = shape
    m = solid.reshape(nz, ny, nx)
    e = G.velocity_set(stencil)
    links = []
    for d in range(1, len(e)):
        hit = (m == 0) & (np.roll(m, tuple(-e[d][::-1]), (0, 1, 2)) != 0)
        lk = np.zeros(int(hit.sum()), G.LINK_DTYPE)
        lk["node"], lk["dir"], lk["bc"], lk["body"], lk["q"] = np.flatnonzero(hit), d, bc, body, q
        links.append(lk)
    links = np.concatenate(links)
    links = links[np.lexsort((links["dir"], links["node"]))]
    return G.Geometry(stencil, nx, ny, nz, (True, True, True), solid, links, (False, False), None, {})


@pytest.mark.parametrize("cfg_g", [0.0, 0.02])
@pytest.mark.parametrize("stencil", [G.D2Q9, G.D3Q19])
def test_fp64_read_out_of_domains_with_weak_and_strong_forces(L, stencil, cfg_g):
    """rho and u of a batch's domains from their own populations, forces inside
    and beyond the grid's (|g| > rho0 / 512) side by side, whatever the lattice's
    own unused force is: 64 eps, as above."""
    forces = [(0.0, 0.0, 0.0), (1e-4, -3e-5, 2e-5), (0.01, -0.004, 0.003), (0.0, 0.05, 0.0), (1e-3, 0.0, 0.0)]
    n, nx, D = 7, 19, 2 if stencil == G.D2Q9 else 3
    shape = (nx, n * len(forces), 1) if D == 2 else (nx, 6, n * len(forces))
    rows = shape[D - 1]
    solid = np.zeros((rows, int(np.prod(shape)) // rows), np.uint8)
    solid[::n] = 1
    solid[n - 1::n] = 1
    geo = _masked(stencil, shape, solid.reshape(-1))
    fl = geo.solid == 0
    lat = L.Lattice(geo, domains=[dict(lo=n * k, n=n, nx=nx, tau=0.7, g=g) for k, g in enumerate(forces)],
                    precision=L.LBM_FP64, tau=0.7, g=(cfg_g, 0.0, 0.0))
    lat.init_equilibrium()
    lat.set_distributions(_state(stencil, geo.N, 1.0, "plain", np.random.default_rng(3)) * fl)
    f = lat.distributions()
    rho, u = lat.moments()
    lat.close()
    e, _ = _weights(stencil)
    g = np.repeat(np.array(forces), geo.N // len(forces), 0).T
    r = np.where(fl, f.sum(0), 1.0)
    ur = ((e.T @ f - 0.5 * g) / r)[:D]
    S = np.abs(f).sum(0) + np.abs(g).sum(0)
    u = u.reshape(D, -1)
    assert np.all(np.abs(rho.reshape(-1) - r)[fl] <= 64 * EPS * S[fl])
    assert np.all(np.abs(u - ur)[:, fl] <= 64 * EPS * (S / r * (1 + np.abs(ur).max(0)))[fl])
