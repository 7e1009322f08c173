"""Steps of a batched launch past the steps whose RF phases are computed at once: the bits of the
same steps taken one launch at a time."""
import numpy as np
import pytest

import iongen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [257, 600, 1100])  # groups of two, four and eight CTAs
def test_batched_steps_do_not_depend_on_the_launch_they_are_in(n):
    import paper_1907_10514_gb300 as it
    counts = [1, 31, 32, 33, 64, 65]

    def sims():
        out = []
        for k in range(len(counts)):
            p = it.make_params(None, Omega=iongen.OMEGA_RF, q=0.2, omega_z=2 * np.pi * 0.1e6, gamma=1e5, T_bath=1e-3,
                               dt=iongen.rf_period_dt(iongen.OMEGA_RF), seed=k, flags=it.IONTRAP_ALLOW_UNSTABLE)
            x = iongen.gaussian_positions(n + k, 30e-6, seed=[n, k])
            out.append(it.Simulation([iongen.Species(iongen.CA40_AMU, 1.0)], np.zeros(n + k, np.uint8), x,
                                     np.zeros((3, n + k)), p))
        return out

    a, b = sims(), sims()
    it.iontrap_step_many([s.handle for s in a], counts)
    for t in range(max(counts)):
        it.iontrap_step_many([s.handle for s in b], [int(t < c) for c in counts])
    for s, r, c in zip(a, b, counts):
        u, w = s.checkpoint(), r.checkpoint()
        assert u[3] == w[3] == c
        for p, q in zip(u[:3], w[:3]):
            assert np.isfinite(p).all() and np.array_equal(p, q)
        s.close(), r.close()
