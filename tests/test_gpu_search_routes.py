"""Which search a handle takes, and the kernels no other test reaches."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

WALL, PER, ABS = 1, 0, 2


def _tube(n, seed, dtype=np.float32, hi=(1, 1, 1), dim=3, bc=(WALL, PER, PER)):
    from paper_1210_8084_gb300 import inputs
    return inputs.cast_state(*inputs.sod_tube(n, seed=seed, hi=hi, dim_pos=dim), dtype, (0, 0, 0), hi, bc)


@pytest.mark.parametrize("prec", [32, 64])
def test_random_partner_variant_searches_nothing(prec):
    """KMC_FLAG_DSMC: no search is chosen, so the scan computes no constants for one."""
    import paper_1210_8084_gb300 as k
    pos, vel = _tube(40_000, 3, np.float32 if prec == 32 else np.float64)
    found = []
    for flags in (0, k.KMC_FLAG_DSMC):
        sim = k.Simulation(k.make_config(dim_pos=3, n_cells=(20, 1, 1), bc=(WALL, PER, PER), lam=1e-3, dt=2e-2,
                                         precision=prec, flags=flags), pos, vel)
        found.append(sim.search()[0])
        sim.close()
    assert found[0] != k.KMC_SEARCH_PARTICLE and found[1] == k.KMC_SEARCH_PARTICLE


def _kinds(k):
    """Handles of binary32 and binary64 on c-bins and, pruned, on finer cells (small and from 2^18 particles on)."""
    yield dict(dim_pos=3, n_cells=(20, 6, 6), hi=(1, .3, .3), lam=1e-3, dt=1e-2, precision=32), 60_000, (1, .3, .3)
    yield dict(dim_pos=3, n_cells=(40, 16, 16), hi=(1, .4, .4), lam=2e-3, dt=5e-3, precision=32), 1 << 18, (1, .4, .4)
    yield dict(dim_pos=3, n_cells=(4, 4, 4), lam=1e-4, dt=2e-2, precision=32), 30_000, (1, 1, 1)
    yield dict(dim_pos=3, n_cells=(16, 5, 5), hi=(1, .3125, .3125), lam=1e-3, dt=1.25e-2, precision=64), 30_000, (1, .3125, .3125)


def test_documented_tile_parameters_are_the_default():
    """A configuration that spells the defaults out, or takes them from kmc_get_info, gets the default search."""
    import paper_1210_8084_gb300 as k
    for base, n, hi in _kinds(k):
        base = dict(base, bc=(WALL, PER, PER), seed=2)
        pos, vel = _tube(n, 6, np.float32 if base["precision"] == 32 else np.float64, hi)
        sim = k.Simulation(k.make_config(**base), pos, vel)
        info, search = sim.info(), sim.search()
        assert search[0] in (k.KMC_SEARCH_FILTER, k.KMC_SEARCH_PAIRS)
        sim.close()
        cap = 1536 if base["precision"] == 32 else 768
        for tile in ((256, cap, 1), (256, 0, 0), (0, cap, 0), (0, 0, 1), (info.tile_threads, info.tile_cap, info.tile_split)):
            sim = k.Simulation(k.make_config(**base, tile_threads=tile[0], tile_cap=tile[1], tile_split=tile[2]), pos, vel)
            again = sim.info()
            assert sim.search() == search and list(again.sub_cells) == list(info.sub_cells), tile
            assert again.kernels_per_step == info.kernels_per_step, tile
            sim.close()
        sim = k.Simulation(k.make_config(**base, tile_threads=128), pos, vel)
        assert sim.search()[0] in (k.KMC_SEARCH_TILE, k.KMC_SEARCH_TILE_PRUNED)
        sim.close()
