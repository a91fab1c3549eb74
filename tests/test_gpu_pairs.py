"""The pair search of binary32 instances (a lane per home, candidates staged and tested
two at a time) finds the same partner for every particle as the search with one
thread per particle: same keys, so the same states bit for bit."""
import numpy as np
import pytest

PER, WALL, ABSORB = 0, 1, 2
pytestmark = pytest.mark.gpu


def _state(seed, n, lo, hi, speed, drift):
    rng = np.random.default_rng(seed)
    lo, hi = np.array(lo, dtype=np.float32), np.array(hi, dtype=np.float32)
    p = (lo + (hi - lo) * rng.random((n, 3), dtype=np.float32)).astype(np.float32)
    p = np.minimum(np.maximum(p, lo), np.nextafter(hi, lo))
    v = (speed * rng.standard_normal((n, 3))).astype(np.float32)
    v[:, 0] += np.float32(drift)
    return p, v


CASES = {
    # dim, cells, boundaries, n, mean free path, dt, drift
    "plane_walls": (2, (40, 40, 1), (WALL, WALL, PER), 40_003, 1e-3, 2e-3, 0.0),
    "plane_periodic": (2, (37, 23, 1), (PER, PER, PER), 30_001, 1e-3, 2e-3, 0.0),
    "plane_four_bins": (2, (4, 4, 1), (PER, PER, PER), 4_000, 1e-3, 2e-2, 0.0),
    "plane_many_pass": (2, (20, 20, 1), (WALL, PER, PER), 60_000, 1e-3, 2e-2, 0.0),
    "plane_cold_stream": (2, (20, 20, 1), (ABSORB, WALL, PER), 40_000, 1e-3, 1e-2, 3.0),
    "slab_one_bin": (3, (300, 1, 1), (WALL, PER, PER), 300_007, 1e-4, 5e-4, 0.0),
    "slab_four_bins": (3, (20, 4, 4), (WALL, PER, PER), 40_000, 1e-3, 4e-3, 0.0),
    "box_periodic": (3, (11, 9, 13), (PER, PER, PER), 30_000, 1e-3, 2e-2, 0.0),
    "plane_wide_reach": (2, (5, 6, 1), (PER, PER, PER), 3_000, 1e-2, 2e-1, 0.0),
}


@pytest.mark.parametrize("name", list(CASES))
def test_pair_search_equals_one_thread_per_particle(name):
    import paper_1210_8084_gb300 as k
    dim, cells, bc, n, lam, dt, drift = CASES[name]
    lo, hi = (0.0, 0.0, 0.0), (1.0, 1.0, 1.0)
    p, v = _state(len(name), n, lo, hi, 1.0 if drift == 0.0 else 0.02, drift)
    out = []
    for flags in (0, k.KMC_FLAG_NO_TILE_SEARCH):
        sim = k.Simulation(k.make_config(dim_pos=dim, n_cells=cells, lo=lo, hi=hi, bc=bc, precision=32, lam=lam, dt=dt,
                                         seed=7, flags=flags), p, v)
        sim.step(3)
        out.append((*sim.state(), sim.moments()[0]))
    for a, b in zip(*out):
        assert np.array_equal(a, b, equal_nan=True)   # NaN: absorbed


def test_pair_search_in_an_uneven_batch():
    """Instances that differ in size take the searches that cost least; each evolves as on its own."""
    import paper_1210_8084_gb300 as k
    base = dict(dim_pos=3, n_cells=(40, 1, 1), lo=(0, 0, 0), hi=(1, 1, 1), bc=(WALL, PER, PER), precision=32)
    ns, insts, P, V = [70_001, 33, 0, 20_000], [], [], []
    for i, n in enumerate(ns):
        p, v = _state(50 + i, n, base["lo"], base["hi"], 1.0, 0.0)
        P.append(p)
        V.append(v)
        insts.append(dict(n=n, lam=1e-3, dt=2e-3, seed=90 + i))
    batch = k.Simulation(k.make_config(**base, instances=insts), np.concatenate(P), np.concatenate(V))
    batch.step(3)
    pb, vb = batch.state()
    off = 0
    for i, n in enumerate(ns):
        if n:
            one = k.Simulation(k.make_config(**base, lam=1e-3, dt=2e-3, seed=90 + i, flags=k.KMC_FLAG_NO_TILE_SEARCH), P[i], V[i])
            one.step(3)
            ps, vs = one.state()
            assert np.array_equal(ps, pb[off:off + n]) and np.array_equal(vs, vb[off:off + n]), i
        off += n
