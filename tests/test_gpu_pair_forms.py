"""The branches of the pair search, each in a handle that kmc_get_search says takes
it: both forms, windows over four periodic c-bins (the one across the box is no
neighbour), and pairs that decide their image themselves (a state set later whose
reach is half the box), all against one thread per particle."""
import numpy as np
import pytest

from test_gpu_pairs import CASES, _state

PER, WALL, ABSORB = 0, 1, 2
pytestmark = pytest.mark.gpu

# name: dim, cells, boundaries, n, mean free path, dt, tested against the closest so far, factor of the speeds set later
BRANCHES = {
    "plane_four_bins": (2, (4, 4, 1), (PER, PER, PER), 40_001, 1e-3, 2.4e-2, True, 1.0),
    "box_four_bins": (3, (4, 4, 4), (PER, PER, PER), 64_000, 1e-4, 1.5e-2, True, 1.0),
    "tube_four_bins": (3, (12, 4, 4), (WALL, PER, PER), 100_003, 1e-4, 1.5e-2, True, 1.0),
    "plane_wide_reach": (2, (5, 6, 1), (PER, PER, PER), 20_003, 1e-3, 2.5e-2, True, 3.0),
    "plane_four_bins_wide": (2, (4, 4, 1), (PER, PER, PER), 40_001, 1e-3, 2.4e-2, True, 2.5),
    "box_wide_reach": (3, (4, 4, 4), (PER, PER, PER), 64_000, 1e-4, 1.5e-2, True, 4.0),
    "slab_wide_reach": (3, (300, 1, 1), (WALL, PER, PER), 300_007, 1e-4, 5e-4, False, 90.0),
}
LISTED = {   # of test_gpu_pairs.py: the form where the pair search is the cheapest
    "plane_walls": False, "plane_periodic": False, "plane_many_pass": True, "plane_cold_stream": True,
    "slab_one_bin": False, "box_periodic": True,
}


@pytest.mark.parametrize("name", list(LISTED))
def test_listed_states_take_the_pair_search(name):
    import paper_1210_8084_gb300 as k
    dim, cells, bc, n, lam, dt, drift = CASES[name]
    p, v = _state(len(name), n, (0, 0, 0), (1, 1, 1), 1.0 if drift == 0.0 else 0.02, drift)
    sim = k.Simulation(k.make_config(dim_pos=dim, n_cells=cells, bc=bc, precision=32, lam=lam, dt=dt, seed=7), p, v)
    assert sim.search() == (k.KMC_SEARCH_PAIRS, k.KMC_FORM_CLOSE if LISTED[name] else 0)
    sim.close()


@pytest.mark.parametrize("name", list(BRANCHES))
def test_branches_equal_one_thread_per_particle(name):
    import paper_1210_8084_gb300 as k
    dim, cells, bc, n, lam, dt, close, factor = BRANCHES[name]
    p, v = _state(7 + len(name), n, (0, 0, 0), (1, 1, 1), 1.0, 0.0)
    out = []
    for flags in (0, k.KMC_FLAG_NO_TILE_SEARCH):
        sim = k.Simulation(k.make_config(dim_pos=dim, n_cells=cells, bc=bc, precision=32, lam=lam, dt=dt, seed=7,
                                         flags=flags | k.KMC_FLAG_RECORD), p, v)
        if flags:
            assert sim.search() == (k.KMC_SEARCH_PARTICLE, 0)
        else:
            assert sim.search() == (k.KMC_SEARCH_PAIRS, k.KMC_FORM_CLOSE if close else 0)
        if factor != 1.0:
            sim.set_state(p, np.float32(factor) * v)
        info = sim.info()
        reach = np.sqrt(info.R2) + 2 * info.vmax * dt
        assert reach > 0.5 if factor != 1.0 else 0.25 < reach < 0.49
        sim.step(2)
        out.append((*sim.partners(), *sim.state(), sim.moments()[0]))
        sim.close()
    assert (out[0][0] >= 0).mean() > 0.5
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def _grazing(rng, x, y, R2, dt, tries=4000):
    """Two particles near (x, y), in binary32, whose path grazes the contact distance:
    criterion 2 met (a^2 - b (r^2 - R^2) >= 0 as rounded), but the distance of closest
    approach r^2 - a^2 / b rounds to more than R^2.  None if no try is one."""
    f = np.float32
    R = np.sqrt(R2)
    t = rng.normal(np.pi / 2, 0.03, tries)
    u = np.stack([np.cos(t), np.sin(t)], 1)             # direction of the relative motion
    w = np.stack([-u[:, 1], u[:, 0]], 1)
    s = rng.uniform(3, 6, tries)[:, None] * R             # path before the closest approach, of 8 R in all
    r = R * w - s * u
    xi = (np.array([x, y]) + 0.5 * r).astype(f)
    xj = (np.array([x, y]) - 0.5 * r).astype(f)
    vi = (4 * u * R / dt).astype(f)
    vj = (-4 * u * R / dt).astype(f)

    def fma(a, b, c):   # the product is exact in binary64; its sum is rounded twice, rarely to another value
        return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(f)
    d, g = xi - xj, vi - vj
    a = fma(d[:, 1], g[:, 1], d[:, 0] * g[:, 0])
    b = fma(g[:, 1], g[:, 1], g[:, 0] * g[:, 0])
    r2 = fma(d[:, 1], d[:, 1], d[:, 0] * d[:, 0])
    disc = fma(a, a, -(b * (r2 - f(R2))))
    d2 = r2 - (a * a) / b
    k = np.flatnonzero((a < 0) & (fma(b, np.full_like(b, dt), a) > 0) & (disc >= 0) & (d2 > f(R2)))
    return None if len(k) == 0 else (xi[k[0]], xj[k[0]], vi[k[0]], vj[k[0]])


def test_pairs_at_the_contact_distance_are_offered_to_both():
    """Isolated pairs whose rounded distance lies just above the contact distance, in a
    handle whose dense half takes the form that tests against the closest so far:
    each is its partner's closest candidate too, so the pair collides."""
    import paper_1210_8084_gb300 as k
    rng = np.random.default_rng(5)
    R, dt = 0.005, 0.01
    R2 = R * R
    lone = [q for q in (_grazing(rng, x, y, R2, dt) for x in np.arange(0.62, 0.97, 0.02) for y in np.arange(0.05, 0.95, 0.07))
            if q is not None]
    assert len(lone) > 100
    p, v = _state(11, 400_000, (0, 0, 0), (0.5, 1, 1), 1.0, 0.0)
    p[:, 2] = v[:, 2] = 0
    n0 = len(p)
    q = np.zeros((2 * len(lone), 3), np.float32)
    w = np.zeros_like(q)
    for i, (xi, xj, vi, vj) in enumerate(lone):
        q[2 * i, :2], q[2 * i + 1, :2], w[2 * i, :2], w[2 * i + 1, :2] = xi, xj, vi, vj
    p, v = np.concatenate([p, q]), np.concatenate([v, w])
    out = []
    for flags in (0, k.KMC_FLAG_NO_TILE_SEARCH):
        sim = k.Simulation(k.make_config(dim_pos=2, n_cells=(20, 20, 1), bc=(WALL, WALL, PER), precision=32, sigma=np.pi * R2,
                                         dt=dt, seed=7, sub_cells=(1, 1, 1), flags=flags | k.KMC_FLAG_RECORD), p, v)
        if not flags:
            assert sim.search() == (k.KMC_SEARCH_PAIRS, k.KMC_FORM_CLOSE)
        sim.step(1)
        out.append((*sim.partners(), *sim.state()))
        sim.close()
    mate = np.arange(2 * len(lone)) ^ 1
    assert (out[1][0][n0:] - n0 == mate).mean() > 0.9   # one thread per particle: both sides
    for a, b in zip(*out):
        assert np.array_equal(a, b)
