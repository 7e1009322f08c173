"""Minimisation in one launch (row-persistent handles): every cluster size and its edges, the
grid above it, and the stop at the tolerance, against the oracle's iterations."""
import numpy as np
import pytest

import iongen
import oracle

pytestmark = pytest.mark.gpu

OMEGA = iongen.OMEGA_RF
DT = 5e-8
DMAX = 5e-7
ITERS = 25


def _case(n):
    sp = (np.arange(n) % 4 == 3).astype(np.uint8)
    x = iongen.gaussian_positions(n, 30e-6, seed=[n, 29])
    trap = iongen.Trap(Omega=OMEGA, a=0.0, q=0.2, omega_z=2 * np.pi * 1e5, gamma=0.0, T_bath=0.0,
                       dt=iongen.rf_period_dt(OMEGA))
    return [iongen.CA40, iongen.NH3], sp, x, trap


@pytest.mark.parametrize("n", [1, 2, 31, 32, 63, 64, 127, 128, 129, 256, 257, 432, 433, 1030])
def test_iterations_match_the_oracle(n):
    """The FP32 pair forces are within 1e-5 of the oracle's: each of the 25 moves of at most
    DMAX keeps its direction to that, times the cloud's amplification over them (below 1e2)."""
    import paper_1907_10514_gb300 as it
    species, sp, x, trap = _case(n)
    q, m, qm0 = oracle.ion_arrays(species, sp)
    po = oracle.params(trap, qm0, flags=oracle.PSEUDO)
    xo, steps, _ = oracle.minimize(x, q, m, po, DT, DMAX, 0.0, ITERS)
    assert steps == ITERS
    with it.Simulation(species, sp, x, None, it.make_params(trap, flags=it.IONTRAP_PSEUDO)) as s:
        assert s.config()[4] == 5
        iters, fn = s.minimize(ITERS, DMAX, 0.0, DT)
        xg, vg, step, _ = s.state()
        assert iters == ITERS and step == 0 and not vg.any()
        assert np.abs(xg - xo).max() < 1e-3 * ITERS * DMAX
        F = m * oracle.accel(xg, np.zeros_like(xg), q, m, po, 0, 0.0)
        assert abs(fn / np.sqrt((F ** 2).sum()) - 1.0) < 1e-4
        # stopped where it already is: no move, the same |F|
        assert s.minimize(10, DMAX, 1.01 * fn, DT) == (0, fn)
        assert np.array_equal(s.state()[0], xg)
        assert s.minimize(0, DMAX, 0.0, DT) == (0, fn)
