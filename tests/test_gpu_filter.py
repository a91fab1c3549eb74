"""The filtered search (tensor-core filter, then the exact test) against the
oracle's closest candidates and against the search of one thread per particle,
where it can go wrong: runs of homes shorter than a warp, tiles that reach past a
row, windows that wrap, that hold their own image (few periodic c-bins) or end at
walls, one and three filters, each pair once or every window, coordinates far
from the origin, systems small enough to share a group between warps."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

WALL, PER, ABS = 1, 0, 2
# name, n, dim, cells, lo, hi, bc, lam, dt, precision, filtered expected (else one kernel: a particle per thread,
# or pairs of candidates where many meet)
CASES = [
    ("one", 1, 3, (2, 2, 2), (0, 0, 0), (1, 1, 1), (PER, PER, PER), 1e-2, 1e-2, 64, False),
    ("two", 2, 3, (1, 1, 1), (0, 0, 0), (1, 1, 1), (PER, PER, PER), 1e-2, 1e-1, 64, False),
    ("tile_edge", 33, 3, (1, 2, 3), (0, 0, 0), (1, 1, 1), (WALL, PER, PER), 1e-2, 5e-2, 64, False),
    ("images64", 700, 3, (3, 1, 2), (0, 0, 0), (1, 1, 1), (PER, PER, PER), 1e-2, 2e-2, 64, True),
    ("images32", 3001, 3, (1, 2, 3), (0, 0, 0), (1, 1, 1), (PER, PER, PER), 1e-2, 1e-2, 32, True),
    ("four_bins", 4003, 3, (4, 4, 4), (0, 0, 0), (1, 1, 1), (PER, PER, PER), 1e-3, 2e-2, 32, True),
    ("five_bins", 4999, 3, (5, 5, 5), (0, 0, 0), (1, 1, 1), (PER, WALL, PER), 1e-3, 2e-2, 64, True),
    ("slab_dense", 20_011, 3, (20, 1, 1), (0, 0, 0), (1, 1, 1), (WALL, PER, PER), 1e-4, 1e-3, 32, True),
    ("slab_thin", 20_000, 3, (100, 1, 1), (0, 0, 0), (1, 1, 1), (WALL, PER, PER), 1e-1, 2e-3, 32, False),
    ("cubic", 30_000, 3, (20, 10, 10), (0, 0, 0), (1, .5, .5), (WALL, PER, PER), 5e-3, 1e-2, 32, True),
    ("cubic_offset", 30_000, 3, (20, 10, 10), (100, -50, 7), (101, -49.5, 7.5), (WALL, PER, PER), 5e-3, 1e-2, 32, True),
    ("absorb", 12_000, 3, (8, 8, 8), (0, 0, 0), (1, 1, 1), (ABS, ABS, ABS), 1e-3, 2e-2, 32, False),
    ("plane", 20_000, 2, (12, 12, 1), (0, 0, 0), (1, 1, 1), (WALL, WALL, PER), 1e-3, 1e-2, 32, False),
    ("plane_wide_contact", 20_000, 2, (16, 16, 1), (0, 0, 0), (1, 1, 1), (PER, WALL, PER), 1e-4, 1e-2, 32, True),
    ("whole_four_bins", 16_003, 3, (4, 4, 4), (0, 0, 0), (1, 1, 1), (PER, PER, PER), 1.0, 2e-3, 32, True),
    ("whole_absorb", 32_000, 3, (5, 5, 5), (0, 0, 0), (1, 1, 1), (ABS, ABS, ABS), 1.0, 2e-3, 32, True),
    ("whole_plane", 20_000, 2, (10, 10, 1), (0, 0, 0), (1, 1, 1), (WALL, PER, PER), 10.0, 1e-3, 32, True),
    ("plane_one_bin", 900, 2, (1, 3, 1), (0, 0, 0), (1, 1, 1), (PER, PER, PER), 1e-2, 1e-2, 64, True),
    ("no_contact", 5000, 3, (4, 4, 4), (0, 0, 0), (1, 1, 1), (WALL, WALL, WALL), 1e30, 1e-2, 64, True),
]


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_filtered_search_matches_oracle_and_per_particle_search(case):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import oracle
    import paper_1210_8084_gb300 as k
    from paper_1210_8084_gb300 import inputs
    name, n, dim, cells, lo, hi, bc, lam, dt, prec, filtered = case
    pos, vel = inputs.sod_tube(n, seed=31, lo=lo, hi=hi, split=0.5 * (lo[0] + hi[0]), dim_pos=dim)
    if bc[0] == PER:
        pos[:, 0] = np.where(pos[:, 0] >= hi[0], lo[0], pos[:, 0])
    dtype = np.float32 if prec == 32 else np.float64
    pos, vel = inputs.cast_state(pos, vel, dtype, lo, hi, bc)
    out, kernels = [], []
    for flags in (0, k.KMC_FLAG_NO_TILE_SEARCH):
        sim = k.Simulation(k.make_config(dim_pos=dim, n_cells=cells, lo=lo, hi=hi, bc=bc, lam=lam, dt=dt, seed=3,
                                         precision=prec, flags=flags | k.KMC_FLAG_RECORD,
                                         sub_cells=(1, 1, 1) if name.startswith("whole") else (0, 0, 0)), pos, vel)
        kernels.append(sim.info().kernels_per_step)
        sim.step(1)
        first = sim.partners()
        sim.step(2)
        out.append((first, sim.partners(), sim.state()))
        sim.close()
    assert kernels[0] - kernels[1] == int(filtered)   # operands and search, or one search
    (f0, l0, s0), (f1, l1, s1) = out
    vol = np.prod([hi[d] - lo[d] for d in range(dim)])
    P = oracle.make_params(dim, cells, lo, hi, bc, R2=oracle.contact_R2(lam, 0.0, n / vol), dt=dt, seed=3, step=0,
                           decide32=prec == 32)
    best = oracle.best_partners(P, pos.astype(np.float64), vel.astype(np.float64))
    if n > 1000 and lam < 1:
        assert (best >= 0).mean() > 0.02
    assert np.array_equal(f0[0], best)
    for a, b in ((f0, f1), (l0, l1), (s0, s1)):   # NaN: absorbed particles
        assert np.array_equal(a[0], b[0], equal_nan=a[0].dtype.kind == "f")
        assert np.array_equal(a[1], b[1], equal_nan=a[1].dtype.kind == "f")


def test_filtered_and_per_particle_instances_share_a_handle():
    """Instances of one handle that take different searches (their particles share
    tiles and groups at the borders) evolve as separate runs."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_1210_8084_gb300 as k
    from paper_1210_8084_gb300 import inputs
    bc = (WALL, PER, PER)
    ns, lams = [9_001, 15, 12_345, 2_003], [1e-1, 1e-3, 1e-4, 1.0]
    base = dict(dim_pos=3, n_cells=(60, 1, 1), bc=bc, precision=32)
    insts, P, V = [], [], []
    for i, (n, lam) in enumerate(zip(ns, lams)):
        p, v = inputs.cast_state(*inputs.sod_tube(n, seed=60 + i), np.float32, (0, 0, 0), (1, 1, 1), bc)
        P.append(p)
        V.append(v)
        insts.append(dict(n=n, lam=lam, dt=2e-3, seed=70 + i))
    batch = k.Simulation(k.make_config(**base, instances=insts), np.concatenate(P), np.concatenate(V))
    assert batch.info().kernels_per_step == 7   # one thread per particle, operands, filtered search; then four more
    batch.step(4)
    pb, vb = batch.state()
    off = 0
    for i, inst in enumerate(insts):
        plain = k.Simulation(k.make_config(**base, lam=inst["lam"], dt=inst["dt"], seed=inst["seed"]), P[i], V[i])
        plain.step(4)
        pp, vp = plain.state()
        assert np.array_equal(pp, pb[off:off + ns[i]]) and np.array_equal(vp, vb[off:off + ns[i]]), i
        plain.close()
        off += ns[i]
    batch.close()


FINE_ROWS = [
    # name, n, dim, cells, hi, bc, lam, search cells per c-bin
    ("few_per_bin", 1 << 18, 3, (40, 16, 16), (1, .4, .4), (WALL, PER, PER), 2e-3, [1, 1, 5]),
    ("many_per_bin", (1 << 18) + 7, 3, (24, 8, 6), (1, 8 / 24, 6 / 24), (WALL, WALL, PER), 2e-2, [2, 2, 8]),
    ("plane", 300_001, 2, (60, 60, 1), (1, 1, 1), (PER, WALL, PER), 5e-2, [1, 8, 1]),
    ("small", (1 << 18) - 1, 3, (40, 16, 16), (1, .4, .4), (WALL, PER, PER), 2e-3, [2, 2, 2]),
]


@pytest.mark.parametrize("case", FINE_ROWS, ids=[c[0] for c in FINE_ROWS])
def test_rows_of_finer_cells_do_not_change_results(case):
    """Pruned instances from 2^18 particles on: rows of search cells finer than half
    c-bins, the candidates and states those of one thread per particle."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_1210_8084_gb300 as k
    from paper_1210_8084_gb300 import inputs
    name, n, dim, cells, hi, bc, lam, sub = case
    lo = (0, 0, 0)
    pos, vel = inputs.sod_tube(n, seed=5, lo=lo, hi=hi, split=0.5, dim_pos=dim)
    pos[:, 0] = np.where(pos[:, 0] >= hi[0], lo[0], pos[:, 0])
    pos, vel = inputs.cast_state(pos, vel, np.float32, lo, hi, bc)
    out = []
    for flags in (0, k.KMC_FLAG_NO_TILE_SEARCH):
        sim = k.Simulation(k.make_config(dim_pos=dim, n_cells=cells, lo=lo, hi=hi, bc=bc, lam=lam, dt=0.2 / cells[0], seed=3,
                                         precision=32, flags=flags | k.KMC_FLAG_RECORD), pos, vel)
        if not flags:
            assert sim.info().tile_prune == 1 and list(sim.info().sub_cells) == sub
        sim.step(2)
        out.append((*sim.partners(), *sim.state(), sim.moments()[0]))
        sim.close()
    assert (out[0][0] >= 0).mean() > 0.01
    for a, b in zip(*out):
        assert np.array_equal(a, b)
