"""The random-partner variant with a thread, a warp or a block per collision cell
(the launch picks by the mean number of particles per cell) against the oracle,
which applies the candidates one after another: cells where almost every pair of
candidates names a common particle, several batches per cell, both precisions."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

WALL, PER = 1, 0


@pytest.mark.parametrize("n,nc,prec,lam,dt", [
    (20, 1, 64, 1e-2, 0.5),        # one warp per cell, far more candidates than particles
    (300, 1, 32, 1e-2, 0.2),       # one block, chains of dependent candidates
    (999, 200, 64, 1e-2, 1e-2),    # one thread per cell, cells of 0 to some particles
    (4001, 100, 32, 1e-3, 5e-3),   # a warp per cell
    (30_011, 13, 64, 1e-3, 1e-2),  # a block per cell, many batches
    (30_011, 200, 32, 1e-3, 1e-3),
])
def test_dsmc_cells_follow_the_sequence(n, nc, prec, lam, dt):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import oracle
    import paper_1210_8084_gb300 as k
    from paper_1210_8084_gb300 import inputs
    lo, hi, bc, cells = (0, 0, 0), (1, 1, 1), (WALL, PER, PER), (nc, 1, 1)
    pos, vel = inputs.sod_tube(n, seed=17)
    pos, vel = inputs.cast_state(pos, vel, np.float32 if prec == 32 else np.float64, lo, hi, bc)
    sim = k.Simulation(k.make_config(dim_pos=3, n_cells=cells, lo=lo, hi=hi, bc=bc, lam=lam, dt=dt, seed=23,
                                     precision=prec, flags=k.KMC_FLAG_DSMC), pos, vel)
    sim.step(1)
    _, vd = sim.state()
    glob = sim.moments()[2]
    sim.close()
    P = oracle.make_params(3, cells, lo, hi, bc, R2=oracle.contact_R2(lam, 0.0, n), dt=dt, seed=23, step=0,
                           decide32=prec == 32)
    _, v, collided, acc = oracle.dsmc_step(P, pos.astype(np.float64), vel.astype(np.float64))
    assert acc > n // 50
    assert glob[0, 6] * 2 == collided.sum()
    err = np.abs(vd - v) / (np.linalg.norm(v, axis=1)[:, None] + 1e-300)
    # the two sides' sin and cos of the direction may differ in the last place; each
    # of a particle's collisions passes its own on, and binary32 rounds after each
    per = 2 * acc / n + 8
    assert err.max() <= per * (1e-13 if prec == 64 else 2.0 ** -22)
