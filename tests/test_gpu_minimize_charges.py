"""Minimisation with charges other than +1 e, on the cluster and on the grid, and iterations that
go on from one launch to the next (after 1000), against the oracle's iterations."""
import numpy as np
import pytest

import iongen
import oracle

pytestmark = pytest.mark.gpu

OMEGA = iongen.OMEGA_RF


def _run(n, charges, iters, dt, dmax):
    import paper_1907_10514_gb300 as it
    species = [iongen.Species(iongen.CA40_AMU, charges[0]), iongen.Species(iongen.NH3_AMU, charges[1])]
    sp = (np.arange(n) % 4 == 3).astype(np.uint8)
    x = iongen.gaussian_positions(n, 30e-6, seed=[n, 41])
    trap = iongen.Trap(Omega=OMEGA, a=0.0, q=0.2, omega_z=2 * np.pi * 1e5, gamma=0.0, T_bath=0.0,
                       dt=iongen.rf_period_dt(OMEGA))
    q, m, qm0 = oracle.ion_arrays(species, sp)
    po = oracle.params(trap, qm0, flags=oracle.PSEUDO)
    xo, steps, _ = oracle.minimize(x, q, m, po, dt, dmax, 0.0, iters)
    assert steps == iters
    with it.Simulation(species, sp, x, None,
                       it.make_params(trap, flags=it.IONTRAP_PSEUDO | it.IONTRAP_ALLOW_UNSTABLE)) as s:
        assert s.config()[4] == 5
        done, fn = s.minimize(iters, dmax, 0.0, dt)
        xg = s.state()[0]
    F = m * oracle.accel(xg, np.zeros_like(xg), q, m, po, 0, 0.0)
    assert done == iters and abs(fn / np.sqrt((F ** 2).sum()) - 1.0) < 1e-4
    return x, xo, xg


@pytest.mark.parametrize("n", [30, 200, 432, 433, 900])
@pytest.mark.parametrize("charges", [(1.0, 2.0), (2.0, 2.0), (1.0, 0.5)])
def test_charged_species(n, charges):
    """As for +1 e: the FP32 pair forces are within 1e-5 of the oracle's, and each of the 25 moves
    of at most dmax keeps its direction to that, times the cloud's amplification (below 1e2)."""
    iters, dmax = 25, 5e-7
    _, xo, xg = _run(n, charges, iters, 5e-8, dmax)
    assert np.abs(xg - xo).max() < 1e-3 * iters * dmax


@pytest.mark.parametrize("n", [100, 500])
def test_iterations_go_on_in_the_next_launch(n):
    """A slow descent (dt = 50 ps, no move near the limit): positions follow x0 + a t^2 / 2 over a
    fraction of the ions' spacing, within 1e-5 of the force times ten for that motion.  Starting the
    last 25 of 1025 iterations from rest would lose 5% of the displacement."""
    x, xo, xg = _run(n, (1.0, 1.0), 1025, 5e-11, 1e-6)
    moved = np.abs(xo - x)
    assert moved.max() < 5e-6
    assert np.sqrt(((xg - xo) ** 2).sum() / (moved ** 2).sum()) < 1e-4
