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
