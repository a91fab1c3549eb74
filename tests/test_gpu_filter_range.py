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


@pytest.mark.parametrize("prec,length,time", [
    (64, 2.0 ** -100, 1.0), (64, 2.0 ** -70, 1.0), (64, 2.0 ** -62, 1.0), (64, 2.0 ** 66, 1.0), (64, 2.0 ** 100, 1.0),
    (64, 2.0 ** 180, 1.0), (64, 1.0, 2.0 ** -180), (64, 1.0, 2.0 ** 180), (64, 2.0 ** 80, 2.0 ** 90),
    (64, 2.0 ** -39, 2.0 ** 30), (64, 2.0 ** 39, 2.0 ** -30),
    (32, 2.0 ** -30, 2.0 ** -30), (32, 2.0 ** 40, 2.0 ** 40),
])
def test_units_of_length_and_time(prec, length, time):
    """Powers of two as units: the run of the same state in units of 1, scaled, bit for bit.
    Binary64 states whose squares leave binary32's range take one thread per particle."""
    import paper_1210_8084_gb300 as k
    from paper_1210_8084_gb300 import inputs
    n, bc = 20_003, (WALL, PER, PER)
    dtype = np.float32 if prec == 32 else np.float64
    pos, vel = inputs.cast_state(*inputs.sod_tube(n, seed=8), dtype, (0, 0, 0), (1, 1, 1), bc)
    out = []
    for u, t in ((1.0, 1.0), (length, time)):
        sim = k.Simulation(k.make_config(dim_pos=3, n_cells=(20, 1, 1), hi=(u, u, u), bc=bc, sigma=u * u / (1e-4 * n), dt=1e-3 * t,
                                         seed=3, precision=prec, flags=k.KMC_FLAG_RECORD), (pos * u).astype(dtype),
                           (vel * (u / t)).astype(dtype))
        fits = prec == 32 or (2.0 ** -40 < u < 2.0 ** 40 and 2.0 ** -50 < t < 2.0 ** 50)
        assert sim.search()[0] == (k.KMC_SEARCH_FILTER if fits else k.KMC_SEARCH_PARTICLE)
        sim.step(3)
        p, v = sim.state()
        out.append((*sim.partners(), p / dtype(u), v / dtype(u / t)))
        sim.close()
    assert (out[0][1] >= 0).mean() > 0.1
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prec,speed", [(32, 1e15), (64, 1e15), (64, 1e34), (64, 1e45), (64, 1e100)])
def test_one_particle_far_faster_than_the_rest(prec, speed):
    """A displacement of 10^12 boxes and more: windows and margins grow (where a speed leaves
    binary32's range every pair passes the filter), no other particle's pairs are lost."""
    import paper_1210_8084_gb300 as k
    from paper_1210_8084_gb300 import inputs
    n, bc = 4_001, (WALL, PER, PER)
    dtype = np.float32 if prec == 32 else np.float64
    pos, vel = inputs.cast_state(*inputs.sod_tube(n, seed=9), dtype, (0, 0, 0), (1, 1, 1), bc)
    cfg = k.make_config(dim_pos=3, n_cells=(20, 1, 1), bc=bc, lam=1e-4, dt=1e-3, seed=3, precision=prec)
    out = []
    for flags in (0, k.KMC_FLAG_NO_TILE_SEARCH):
        cfg.flags = k.KMC_FLAG_RECORD | flags
        sim = k.Simulation(cfg, pos, vel)
        assert sim.search()[0] == (k.KMC_SEARCH_PARTICLE if flags else k.KMC_SEARCH_FILTER)
        fast = vel.copy()
        fast[5] = speed * np.array([1.0, -2.0, 0.3])
        sim.set_state(pos, fast)
        sim.step(1)
        out.append((*sim.partners(), *sim.state()))
        sim.close()
    assert (out[1][0] >= 0).mean() > 0.3
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prec,unit", [(64, 2.0 ** -70), (64, 2.0 ** 30), (64, 2.0 ** 100), (32, 2.0 ** 30)])
def test_partner_call_in_other_units(prec, unit):
    torch = pytest.importorskip("torch")
    import paper_1210_8084_gb300 as k
    from paper_1210_8084_gb300 import inputs
    n, bc = 10_007, (WALL, PER, PER)
    dtype = np.float32 if prec == 32 else np.float64
    pos, vel = inputs.cast_state(*inputs.sod_tube(n, seed=8), dtype, (0, 0, 0), (1, 1, 1), bc)
    out = []
    for u in (1.0, unit):
        cfg = k.make_config(dim_pos=3, n_cells=(20, 1, 1), hi=(u, u, u), bc=bc, sigma=u * u / (1e-4 * n), dt=1e-3 * u, precision=prec)
        p, v = torch.from_numpy((pos * u).astype(dtype)).cuda(), torch.from_numpy(vel).cuda()
        best = torch.full((n,), -7, dtype=torch.int32, device="cuda")
        assert k.kmc_find_partners_noalloc(cfg, n, p, v, best) == k.KMC_OK
        torch.cuda.synchronize()
        out.append(best.cpu().numpy())
    assert (out[0] >= 0).mean() > 0.3
    assert np.array_equal(*out)


@pytest.mark.parametrize("offset", [1e3, 1e6, 1e9])
def test_binary64_box_far_from_the_origin(offset):
    """The pairs of one thread per particle, and (the margins do not grow with the offset) about the
    search's time at the origin: bounds of binary32 coordinates let nearly every pair pass from 10^6 on."""
    import paper_1210_8084_gb300 as k
    from paper_1210_8084_gb300 import inputs
    n, bc = 200_000, (WALL, PER, PER)
    ms, out = [], []
    for off, flags in ((0.0, 0), (offset, 0), (offset, k.KMC_FLAG_NO_TILE_SEARCH)):
        lo, hi = (off,) * 3, (off + 1,) * 3
        pos, vel = inputs.cast_state(*inputs.sod_tube(n, seed=4, lo=lo, hi=hi, split=off + 0.5), np.float64, lo, hi, bc)
        sim = k.Simulation(k.make_config(dim_pos=3, n_cells=(200, 1, 1), lo=lo, hi=hi, bc=bc, lam=1e-3, dt=1e-3, seed=3,
                                         precision=64, flags=flags | k.KMC_FLAG_RECORD), pos, vel)
        assert sim.search()[0] == (k.KMC_SEARCH_PARTICLE if flags else k.KMC_SEARCH_FILTER)
        ms.append(min(sim.step_profiled(1)["search"] for _ in range(5)))
        out.append((*sim.partners(), *sim.state()))
        sim.close()
    assert (out[1][1] >= 0).mean() > 0.1
    for a, b in zip(out[1], out[2]):
        assert np.array_equal(a, b)
    assert ms[1] < 1.5 * ms[0], ms
