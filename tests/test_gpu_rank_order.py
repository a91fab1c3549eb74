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


@pytest.mark.parametrize("order", ["mixed", "by_cell", "few_far", "parts"])
@pytest.mark.parametrize("cells,counts", [(3, [192, 193, 300]), (40, 500), (5, [4096, 700, 0, 4097, 2000]), (3, [16384, 16383, 9000])],
                         ids=str)
def test_order_in_cells(cells, counts, order):
    import paper_1210_8084_gb300 as k
    cell = _cells(order, cells, counts)
    n = len(cell)
    sim = _sim(k, cells, cell)
    perm = sim.perm()
    where = sim.cell_keys()[perm]
    assert np.array_equal(np.sort(perm), np.arange(n))
    assert np.all(np.diff(where) >= 0)
    for c in range(cells):
        assert np.all(np.diff(perm[where == c]) > 0) or np.count_nonzero(where == c) > 16384
    sim.close()


def test_ids_in_cell_order_take_no_longer():
    """A state generated cell by cell: a cell's ids are a narrow range of the instance's."""
    import paper_1210_8084_gb300 as k
    ms = {}
    for order in ("mixed", "by_cell"):
        sim = _sim(k, 2000, _cells(order, 2000, 2000))
        ms[order] = min(sim.step_profiled(1)["scatter"] for _ in range(5))
        sim.close()
    assert ms["by_cell"] < 2.0 * ms["mixed"], ms


@pytest.mark.parametrize("mean,launches", [(40, 0), (100, 0), (200, 1), (2000, 2)])
def test_small_cells_are_not_ranked(mean, launches):
    """Cells of less than some two hundred particles are put in order by the moving pass."""
    import paper_1210_8084_gb300 as k
    sim = _sim(k, 50, _cells("mixed", 50, mean), flags=k.KMC_FLAG_DSMC)
    assert sim.info().kernels_per_step == 5 + launches   # collisions, move, scan, two scatter passes, ranking
    sim.close()
