"""Three periodic c-bins: all are neighbours of one another, so the pair whose
shortest separation crosses a whole c-bin is a candidate like any other (every
search against the oracle, and one constructed pair)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

WALL, PER = 1, 0


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_pair_across_a_c_bin(axis, prec):
    """x = 0.33 and 0.72, closing in: 0.39 apart directly (0.61 around the box), in c-bins 0 and 2."""
    import paper_1210_8084_gb300 as k
    dtype = np.float32 if prec == 32 else np.float64
    pos = np.full((2, 3), 0.5, dtype)
    vel = np.zeros((2, 3), dtype)
    pos[:, axis], vel[:, axis] = (0.33, 0.72), (30.0, -30.0)
    for sub in ((6, 6, 6), (1, 1, 1), (2, 5, 3)):
        sim = k.Simulation(k.make_config(dim_pos=3, n_cells=(3, 3, 3), bc=(PER, PER, PER), sigma=np.pi * 0.03 ** 2, dt=0.0068, precision=prec,
                                         sub_cells=sub, flags=k.KMC_FLAG_RECORD), pos, vel)
        sim.step(1)
        best, partner = sim.partners()
        sim.close()
        assert list(best) == [1, 0] and list(partner) == [1, 0], sub


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("dim,cells,bc,dt", [(3, (3, 3, 3), (PER, PER, PER), 0.05), (3, (3, 4, 3), (PER, PER, WALL), 0.04),
                                             (2, (3, 3, 1), (PER, PER, PER), 0.06), (3, (3, 1, 2), (PER, PER, PER), 0.045)])
def test_searches_match_the_oracle(dim, cells, bc, dt, prec):
    import oracle
    import paper_1210_8084_gb300 as k
    n, R = 1_500, 0.03
    dtype = np.float32 if prec == 32 else np.float64
    rng = np.random.default_rng(5)
    pos, vel = (0.999 * rng.random((n, 3))).astype(dtype), rng.standard_normal((n, 3)).astype(dtype)
    if dim == 2:
        pos[:, 2] = 0
    P = oracle.make_params(dim, cells, (0, 0, 0), (1, 1, 1), bc, R2=oracle.contact_R2(0.0, np.pi * R * R, n), dt=dt, seed=1, step=0,
                           decide32=prec == 32)
    best = oracle.best_partners(P, pos.astype(np.float64), vel.astype(np.float64))
    assert (best >= 0).mean() > 0.2
    for opt in (dict(), dict(flags=k.KMC_FLAG_NO_TILE_SEARCH), dict(flags=k.KMC_FLAG_STAGED_SEARCH), dict(tile_threads=128)):
        for sub in ((0, 0, 0), (5, 4, 6), (1, 1, 1)):
            opts = dict(opt, flags=opt.get("flags", 0) | k.KMC_FLAG_RECORD)
            sim = k.Simulation(k.make_config(dim_pos=dim, n_cells=cells, bc=bc, sigma=np.pi * R * R, dt=dt, seed=1, precision=prec,
                                             sub_cells=sub, **opts), pos, vel)
            sim.step(1)
            got, _ = sim.partners()
            sim.close()
            assert np.array_equal(got, best), (opt, sub)
