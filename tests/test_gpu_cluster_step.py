"""The cluster launch of small row-persistent simulations gives the bits of the grid launch of
the same shape.  Launches with a wait limit of their own (iontrap_test_stall) take the grid."""
import numpy as np
import pytest

import iongen

pytestmark = pytest.mark.gpu


def _handle(it, n, charges, laser, flags):
    rng = np.random.default_rng([n, 17])
    x = iongen.gaussian_positions(n, 20e-6, seed=[n, 3])
    v = rng.normal(size=(3, n))
    sp = (np.arange(n) % 3 == 2).astype(np.uint8)
    species = [iongen.Species(iongen.CA40_AMU, charges[0]), iongen.Species(iongen.NH3_AMU, charges[1])]
    p = it.make_params(None, Omega=iongen.OMEGA_RF, q=0.2, omega_z=2 * np.pi * 0.1e6, gamma=1e5, T_bath=1e-3,
                       dt=iongen.rf_period_dt(iongen.OMEGA_RF), seed=n, flags=flags | it.IONTRAP_ALLOW_UNSTABLE)
    s = it.Simulation(species, sp, x, v, p)
    if laser:
        s.set_params(p, [(1e5, 1e-3, (3e5, -2e5, 1e5)), (0.0, 0.0, (0.0, 1e5, 0.0))])
    return s


# edges of the cluster sizes (12, 13, 28, 29, 84, 85, 432 | 433), ions not a multiple of four,
# parts of 4 entries up to a chunk, one and two ions per thread, more parts than ions
@pytest.mark.parametrize("n,cfg", [
    (2, (256, 1, 1)), (5, (256, 1, 2)), (12, (256, 1, 5)), (13, (512, 1, 4)), (28, (256, 2, 9)), (29, (256, 1, 7)),
    (84, (512, 2, 40)), (85, (256, 1, 1)), (130, (256, 1, 64)), (321, (256, 1, 3)), (431, (256, 1, 32)),
    (432, (512, 1, 30)), (433, (256, 1, 3)), (300, (256, 1, 85)),
])
@pytest.mark.parametrize("charges,laser,pseudo", [((1.0, 1.0), True, False), ((1.0, 2.0), False, False),
                                                  ((1.0, 1.0), False, True)])
def test_cluster_steps_are_the_grid_steps_bit_for_bit(n, cfg, charges, laser, pseudo):
    import paper_1907_10514_gb300 as it
    got = []
    for grid in (False, True):
        with _handle(it, n, charges, laser, it.IONTRAP_PSEUDO if pseudo else 0) as s:
            s.set_config(cfg[0], cfg[1], 1, cfg[2], 5, 0, 0)
            if grid:
                it.iontrap_test_stall(s.handle, 2_000_000_000, -1, 0)
            for k in (1, 2, 45):
                s.step(k)
            x, v, a, step = s.checkpoint()
            assert step == 48
            s.step(3)
            got.append((x, v, a, s.state()[0]))
    for u, w in zip(*got):
        assert np.isfinite(u).all() and np.array_equal(u, w)
