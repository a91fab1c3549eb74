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
