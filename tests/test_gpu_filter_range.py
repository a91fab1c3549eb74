"""The filtered search where its 16- and 32-bit operands could leave their range:
contact distances far beyond the box, and boxes in units far from 1."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

WALL, PER, ABS = 1, 0, 2


def _partners(k, cfg, pos, vel, steps, want):
    """Closest candidates and partners of every step and the last state, with and without the filtered search."""
    out = []
    for flags in (0, k.KMC_FLAG_NO_TILE_SEARCH):
        cfg.flags = k.KMC_FLAG_RECORD | flags
        sim = k.Simulation(cfg, pos, vel)
        if not flags:
            assert sim.search()[0] == want
        got = []
        for _ in range(steps):
            sim.step(1)
            got += [*sim.partners()]
        out.append((*got, *sim.state()))
        sim.close()
    return out


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("lam", [1e-4, 1e-6, 1e-8, 1e-12, 1e-30])
@pytest.mark.parametrize("cells,bc", [((4, 4, 4), (WALL, PER, PER)), ((6, 7, 1), (WALL, WALL, WALL))], ids=["mixed", "walls"])
def test_contact_distance_beyond_the_box(prec, lam, cells, bc):
    """R from about the box's length to far beyond it: every approaching pair is within it."""
    import paper_1210_8084_gb300 as k
    from paper_1210_8084_gb300 import inputs
    n = 3_001
    dtype = np.float32 if prec == 32 else np.float64
    pos, vel = inputs.cast_state(*inputs.sod_tube(n, seed=12), dtype, (0, 0, 0), (1, 1, 1), bc)
    cfg = k.make_config(dim_pos=3, n_cells=cells, bc=bc, lam=lam, dt=2e-2, seed=3, precision=prec)
    out = _partners(k, cfg, pos, vel, 2, k.KMC_SEARCH_PAIRS if (prec, lam, cells[2]) == (32, 1e-4, 1) else k.KMC_SEARCH_FILTER)
    assert (out[1][0] >= 0).mean() > 0.3
    for a, b in zip(*out):
        assert np.array_equal(a, b)
