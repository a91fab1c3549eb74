"""Order of particles inside large search cells (ranked by a block per cell): the
sort permutation is (cell, id) at the sizes where the kernel starts, fills its
shared memory, hands over to the second launch, and for cells whose ids are a
narrow range or clash in few buckets."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

WALL, PER = 1, 0


@pytest.mark.parametrize("cells,counts", [
    (1, [64]), (1, [65]), (1, [4096]), (1, [4097]), (1, [16384]),
    (2, [4096, 31]), (3, [65, 0, 2000]), (4, [1, 64, 16383, 5000]), (2, [16385, 300]),
], ids=str)
@pytest.mark.parametrize("order", ["mixed", "by_cell", "reversed"])
def test_large_cells_are_in_id_order(cells, counts, order):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_1210_8084_gb300 as k
    n = sum(counts)
    rng = np.random.default_rng(n)
    cell = np.repeat(np.arange(cells), counts)
    if order == "mixed":
        rng.shuffle(cell)
    elif order == "reversed":
        cell = cell[::-1].copy()
    pos = rng.random((n, 3))
    pos[:, 0] = (cell + 0.1 + 0.8 * pos[:, 0]) / cells
    pos = pos.astype(np.float32)
    vel = rng.normal(size=(n, 3)).astype(np.float32)
    sim = k.Simulation(k.make_config(dim_pos=3, n_cells=(cells, 1, 1), bc=(WALL, PER, PER), lam=1e6, dt=1e-6, seed=1,
                                     precision=32, sub_cells=(1, 1, 1)), pos, vel)
    for _ in range(2):   # the initial sort, then the sort of a step that hardly moves anything
        perm = sim.perm()
        where = sim.cell_keys()[perm]
        assert np.array_equal(np.sort(perm), np.arange(n))
        assert np.all(np.diff(where) >= 0)
        for c in range(cells):
            ids = perm[where == c]
            if len(ids) <= 16384:
                assert np.all(np.diff(ids) > 0)
        sim.step(1)
    sim.close()
