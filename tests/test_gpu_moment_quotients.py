"""Quotients of the derived moments (by a reciprocal and one step on the residual)
are those of a division, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n,cells", [(32, 3_000_000, 100_000), (64, 1_000_000, 250_000), (64, 2_000_000, 3)])
def test_mean_velocities_are_correctly_rounded(prec, n, cells):
    import paper_1210_8084_gb300 as k
    rng = np.random.default_rng(cells)
    dtype = np.float32 if prec == 32 else np.float64
    pos = rng.random((n, 3)).astype(dtype) * dtype(0.999)
    pos[:, 0] **= 3   # counts from a few to many
    vel = (rng.standard_normal((n, 3)) * 10.0 ** rng.uniform(-6, 6, (n, 1))).astype(dtype)
    sim = k.Simulation(k.make_config(dim_pos=3, n_cells=(cells, 1, 1), bc=(1, 0, 0), lam=1e3, dt=1e-12, precision=prec,
                                     flags=k.KMC_FLAG_RADIAL_MOMENT, radial_center=(0.5, 0.5, 0.5)), pos, vel)
    raw, der, _ = sim.moments()
    rad = sim.radial()
    sim.close()
    full = raw[:, 0] > 0
    count = raw[full, 0]
    assert raw[:, 0].sum() == n
    for c in range(3):
        assert np.array_equal(der[full, 1 + c], raw[full, 1 + c] / count)
    assert np.array_equal(rad[full, 1], rad[full, 0] / count)
