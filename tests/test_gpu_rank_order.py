"""The scatter's order inside search cells where ids follow the positions: same
order as for ids without any, in about the same time."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

WALL, PER = 1, 0


def _sim(k, cells, cell, seed=1, flags=0):
    """A state whose particle i lies in slab cell[i], at rest but for small speeds."""
    rng = np.random.default_rng(seed)
    n = len(cell)
    pos = rng.random((n, 3), dtype=np.float32)
    pos[:, 0] = (cell + np.float32(0.1) + np.float32(0.8) * pos[:, 0]) / np.float32(cells)
    vel = rng.standard_normal((n, 3), dtype=np.float32)
    return k.Simulation(k.make_config(dim_pos=3, n_cells=(cells, 1, 1), bc=(WALL, PER, PER), lam=1e6, dt=1e-6, seed=1,
                                      precision=32, sub_cells=(1, 1, 1), flags=flags), pos, vel)


def _cells(order, cells, counts, seed=2):
    rng = np.random.default_rng(seed)
    cell = np.repeat(np.arange(cells), counts)
    if order == "mixed":
        rng.shuffle(cell)
    elif order == "few_far":   # cell by cell, but a few particles of each among the others
        i = rng.permutation(len(cell))[:4 * cells]
        cell[i] = cell[np.roll(i, 1)]
    elif order == "parts":     # several parts, each cell by cell
        cell = np.concatenate([np.sort(c) for c in np.array_split(rng.permutation(cell), 8)])
    return cell


@pytest.mark.parametrize("mean,launches", [(40, 0), (100, 0), (200, 1), (2000, 2)])
def test_small_cells_are_not_ranked(mean, launches):
    """Cells of less than some two hundred particles are put in order by the moving pass."""
    import paper_1210_8084_gb300 as k
    sim = _sim(k, 50, _cells("mixed", 50, mean), flags=k.KMC_FLAG_DSMC)
    assert sim.info().kernels_per_step == 5 + launches   # collisions, move, scan, two scatter passes, ranking
    sim.close()
