"""The state comes back in id order, whole or one array of it, on both sides of the
size where the read-back takes two passes, and with absorbed particles as NaN."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PER, ABS = 0, 2


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("n", [1, 255, 524_287, 524_288, 524_545])
def test_state_comes_back_in_id_order(n, prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_1210_8084_gb300 as k
    dtype = np.float32 if prec == 32 else np.float64
    rng = np.random.default_rng(n)
    pos, vel = rng.random((n, 3)).astype(dtype) * dtype(0.999), rng.normal(size=(n, 3)).astype(dtype)
    gone = rng.random(n) < 0.01
    pos[gone] = np.nan
    vel[gone] = np.nan
    insts = [dict(n=n // 3, lam=1e-3, dt=1e-3), dict(n=n - n // 3, lam=1e-2, dt=1e-3)] if n > 2 else None
    sim = k.Simulation(k.make_config(dim_pos=3, n_cells=(20, 20, 20), bc=(ABS, PER, PER), lam=1e-3, dt=1e-3,
                                     precision=prec, instances=insts), pos, vel)
    p, v = sim.state()
    assert np.array_equal(p, pos, equal_nan=True) and np.array_equal(v, vel, equal_nan=True)
    only = np.zeros_like(vel)
    k.kmc_get_state(sim.h, None, only)
    assert np.array_equal(only, vel, equal_nan=True)
    k.kmc_get_state(sim.h, only, None)
    assert np.array_equal(only, pos, equal_nan=True)
    sim.close()
