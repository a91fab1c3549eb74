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


def test_tile_searches_of_a_mixed_batch():
    """Tile parameters: the plain and the pruned tile search in one launch sequence, each instance as on
    its own with the default searches."""
    import paper_1210_8084_gb300 as k
    hi, cells = (1, 0.5, 0.5), (12, 6, 6)
    ns, lams = [40_000, 30_000, 20_000], [5e-3, 1e-4, 5e-2]
    state = [_tube(n, 200 + i, hi=hi) for i, n in enumerate(ns)]
    insts = [dict(n=n, lam=lam, dt=1e-2, seed=300 + i) for i, (n, lam) in enumerate(zip(ns, lams))]
    base = dict(dim_pos=3, n_cells=cells, hi=hi, bc=(WALL, PER, PER), precision=32)
    batch = k.Simulation(k.make_config(**base, instances=insts, tile_threads=128), np.concatenate([s[0] for s in state]),
                         np.concatenate([s[1] for s in state]))
    assert [batch.search(i)[0] for i in range(3)] == [k.KMC_SEARCH_TILE_PRUNED, k.KMC_SEARCH_TILE, k.KMC_SEARCH_TILE_PRUNED]
    assert batch.info().kernels_per_step == 6   # plain tile search, pruned tile search, move, scan, two scatter passes
    batch.step(3)
    pb, vb = batch.state()
    off = 0
    for i, (p, v) in enumerate(state):
        one = k.Simulation(k.make_config(**base, lam=lams[i], dt=1e-2, seed=300 + i), p, v)
        assert one.search()[0] in (k.KMC_SEARCH_FILTER, k.KMC_SEARCH_PAIRS, k.KMC_SEARCH_PARTICLE)
        one.step(3)
        po, vo = one.state()
        assert np.array_equal(po, pb[off:off + ns[i]]) and np.array_equal(vo, vb[off:off + ns[i]]), i
        off += ns[i]
        one.close()
    batch.close()


@pytest.mark.parametrize("dim", [2, 3])
def test_pruned_tile_search_at_its_own_staging_capacity(dim):
    """tile_split alone keeps the pruned tile search's default capacity (an instance of the kernel of its own)."""
    import paper_1210_8084_gb300 as k
    n, cells, hi, lam, dt = (60_000, (20, 6, 6), (1, .3, .3), 1e-3, 1e-2) if dim == 3 else (200_000, (40, 40, 1), (1, 1, 1), 0.02, 5e-3)
    bc = (WALL, PER, PER) if dim == 3 else (WALL, WALL, PER)
    pos, vel = _tube(n, 21, hi=hi, dim=dim, bc=bc)
    out = []
    for split in (2, 0):
        sim = k.Simulation(k.make_config(dim_pos=dim, n_cells=cells, hi=hi, bc=bc, lam=lam, dt=dt, seed=5, precision=32,
                                         tile_split=split, flags=k.KMC_FLAG_RECORD), pos, vel)
        assert sim.search()[0] == (k.KMC_SEARCH_TILE_PRUNED if split else k.KMC_SEARCH_FILTER)
        assert sim.info().tile_cap == 1888
        sim.step(2)
        out.append((*sim.partners(), *sim.state()))
        sim.close()
    assert (out[0][0] >= 0).mean() > 0.05
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 31, 33, 64, 255, 513])
def test_filtered_search_of_a_few_particles(n):
    """Pruned instances of a batch are filtered at any size: part of a tile, of a group and of a warp's share."""
    import oracle
    import paper_1210_8084_gb300 as k
    rng = np.random.default_rng(n)
    cells, bc, R, dt = (6, 6, 1), (PER, WALL, PER), 0.08, 0.05
    pos, vel = rng.random((n, 3), dtype=np.float32), rng.standard_normal((n, 3), dtype=np.float32)
    if n <= 9:
        pos[:, :2] = 0.4 + 0.2 * pos[:, :2]   # close enough to meet
    pos[:, 2] = 0
    insts = [dict(n=m, sigma=np.pi * R * R, lam=1.0, dt=dt, seed=4) for m in (n, 0)]
    sim = k.Simulation(k.make_config(dim_pos=2, n_cells=cells, bc=bc, instances=insts, precision=32, flags=k.KMC_FLAG_RECORD),
                       pos, vel)
    assert sim.search(0)[0] == k.KMC_SEARCH_FILTER
    sim.step(1)
    best, _ = sim.partners()
    sim.close()
    P = oracle.make_params(2, cells, (0, 0, 0), (1, 1, 1), bc, R2=oracle.contact_R2(0.0, np.pi * R * R, n), dt=dt, seed=4, step=0,
                           decide32=True)
    assert np.array_equal(best, oracle.best_partners(P, pos.astype(np.float64), vel.astype(np.float64)))


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("n,nc,empty", [(8_003, 4, 9), (8_003, 4, 254), (400, 2, 60)])
def test_random_partner_variant_is_the_same_by_thread_warp_and_block(n, nc, empty, prec):
    """The launch gives a cell a thread, a warp or a block by the mean number of particles; empty instances beside
    the same one lower the mean.  Bit for bit, over cells in which nearly all candidates depend on others."""
    import paper_1210_8084_gb300 as k
    dtype = np.float32 if prec == 32 else np.float64
    pos, vel = _tube(n, 30, dtype)
    base = dict(dim_pos=3, n_cells=(nc, 1, 1), bc=(WALL, PER, PER), precision=prec, flags=k.KMC_FLAG_DSMC)
    one = dict(n=n, lam=1e-3, dt=2e-2, seed=77)
    out = []
    for extra in (0, empty):
        insts = [one] + [dict(n=0, lam=1e-3, dt=2e-2, seed=i) for i in range(extra)]
        cfg = k.make_config(**base, instances=insts) if extra else k.make_config(**base, lam=1e-3, dt=2e-2, seed=77)
        sim = k.Simulation(cfg, pos, vel)
        sim.step(3)
        out.append(sim.state())
        sim.close()
    assert not np.array_equal(out[0][1], vel)
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prec,n,cells", [(32, 400_000, (60, 16, 16)), (32, 2_000_000, (120, 32, 32)), (64, 436_649, (109, 19, 19))])
def test_thin_particles_beside_a_cluster(prec, n, cells):
    """A third of the particles in a hundredth of the box, contact distance and displacement far below a cell: the
    filtered search would walk hundreds of frame blocks for the thin rows (24 times as long as one thread per particle)."""
    import paper_1210_8084_gb300 as k
    rng = np.random.default_rng(3)
    dtype = np.float32 if prec == 32 else np.float64
    hi = np.array([1.0, cells[1] / cells[0], cells[2] / cells[0]])
    pos = rng.random((n, 3)) * 0.9999
    pos[:n // 3] = 0.4 + 0.1 * pos[:n // 3]
    pos, vel = (pos * hi).astype(dtype), rng.standard_normal((n, 3)).astype(dtype)
    R = (0.013 if prec == 32 else 0.004) / cells[0]
    ms = []
    for flags in (0, k.KMC_FLAG_NO_TILE_SEARCH):
        sim = k.Simulation(k.make_config(dim_pos=3, n_cells=cells, hi=tuple(hi), bc=(PER, PER, WALL), sigma=np.pi * R * R,
                                         dt=0.011 / cells[0], seed=1, precision=prec, flags=flags), pos, vel)
        sim.step(1)
        ms.append(min(sim.step_profiled(1)["search"] for _ in range(4)))
        sim.close()
    assert ms[0] < 1.5 * ms[1], ms


@pytest.mark.parametrize("n,dim,cells,hi,R,dt,search", [
    (3_708, 3, (39, 6, 6), (1, 6 / 39, 6 / 39), 0.49, 0.11, 4), (10_860, 2, (85, 8, 1), (1, 8 / 85, 1), 0.022, 0.3, 4),
    (4_254, 3, (29, 6, 6), (1, 6 / 29, 6 / 29), 0.022, 0.13, 4), (2_189, 3, (34, 4, 4), (1, 4 / 34, 4 / 34), 0.03, 0.34, 3)])
def test_small_runs_take_no_longer_than_a_block_per_c_bin(n, dim, cells, hi, R, dt, search):
    """A few thousand particles in hundreds of c-bins: the tile searches' latency beats the filter's (up to 4.9 times)."""
    import paper_1210_8084_gb300 as k
    bc = (PER, PER, WALL)
    pos, vel = _tube(n, 41, hi=hi, dim=dim, bc=bc)
    pos[:, 0] = np.minimum(pos[:, 0], np.nextafter(np.float32(1), np.float32(0)))
    base = dict(dim_pos=dim, n_cells=cells, hi=hi, bc=bc, sigma=np.pi * (R / cells[0]) ** 2, dt=dt / cells[0], seed=1, precision=32)
    ms = []
    for tile in (0, 1534):   # not the default capacity: asks for the tile search
        sim = k.Simulation(k.make_config(**base, tile_cap=tile), pos, vel)
        assert sim.search()[0] == search
        sim.step(1)
        ms.append(min(p["search"] + p["tile"] for p in (sim.step_profiled(1) for _ in range(6))))
        sim.close()
    assert ms[0] < 1.5 * ms[1], ms


def test_partner_call_where_windows_reach_around_the_box():
    """Three periodic c-bins across: a step's reach is half the box, where the pair search decides every pair
    exactly (9 times as long as one thread per particle); the call, without statistics of the state, keeps off it."""
    import torch
    import paper_1210_8084_gb300 as k
    rng = np.random.default_rng(8)
    n, cells = 3_528, (13, 3, 3)
    hi = (1.0, 3 / 13, 3 / 13)
    pos, vel = (0.9999 * rng.random((n, 3)) * hi).astype(np.float32), rng.standard_normal((n, 3), dtype=np.float32)
    R = 0.04 / 13
    base = dict(dim_pos=3, n_cells=cells, hi=hi, bc=(PER, PER, PER), sigma=np.pi * R * R, dt=0.178 / 13, precision=32,
                sub_cells=(2, 3, 2))
    p, v, best = torch.from_numpy(pos).cuda(), torch.from_numpy(vel).cuda(), torch.empty(n, dtype=torch.int32, device="cuda")
    cfg = k.make_config(**base)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ms = []
    for _ in range(6):
        e0.record(torch.cuda.default_stream())
        assert k.kmc_find_partners_noalloc(cfg, n, p, v, best) == k.KMC_OK
        e1.record(torch.cuda.default_stream())
        torch.cuda.synchronize()
        ms.append(e0.elapsed_time(e1))
    sim = k.Simulation(k.make_config(**base, flags=k.KMC_FLAG_NO_TILE_SEARCH), pos, vel)
    sim.step(1)
    direct = min(sim.step_profiled(1)["search"] for _ in range(4))
    sim.close()
    assert min(ms) < 2 * direct + 0.1, (min(ms), direct)
