"""The FP64 form's pair line: forces of every row-block width (1, 2, 4 and 8 ions per lane) and
ragged last blocks against the oracle, with charges of several sizes and signs."""
import numpy as np
import pytest

import iongen
import oracle

pytestmark = pytest.mark.gpu

# a pair's term is within 3 ulp and an ion's sum of N terms within N/2 ulp of its absolute sum;
# the clouds' cancellation stays below 1e3: 1e-12 holds with room at every N here
TOL = 1e-12


@pytest.mark.parametrize("n", [2, 31, 33, 65, 1000, 2048, 2049, 4096, 4097, 8192, 8193])
@pytest.mark.parametrize("unit", [True, False])
def test_fp64_forces_and_two_steps(n, unit):
    import paper_1907_10514_gb300 as it
    rng = np.random.default_rng([n, 23])
    x = iongen.gaussian_positions(n, 30e-6 * max(1.0, n / 512.0) ** (1 / 3), seed=[n, 7])
    sp = rng.integers(0, 3, n).astype(np.uint8)
    species = [iongen.Species(40.0, 1.0), iongen.Species(17.0, 1.0 if unit else 2.0),
               iongen.Species(137.0, 1.0 if unit else -1.0)]
    p = it.make_params(None, precision=it.IONTRAP_PREC_FP64, Omega=iongen.OMEGA_RF, q=0.2, omega_z=2 * np.pi * 1e5,
                       gamma=1e5, T_bath=1e-3, dt=iongen.rf_period_dt(iongen.OMEGA_RF), seed=3,
                       flags=it.IONTRAP_ALLOW_UNSTABLE)
    q, m, _ = oracle.ion_arrays(species, sp)
    idx = np.arange(n) if n <= 4097 else np.unique(np.r_[np.arange(40), rng.integers(0, n, 200), np.arange(n - 40, n)])
    with it.Simulation(species, sp, x, None, p) as s:
        for k in range(2):  # the initial positions, then those two steps on
            f = s.forces()
            ref = oracle.coulomb_accel(s.state()[0], q, m, idx=idx)
            assert np.sqrt(((f[:, idx] - ref) ** 2).sum() / (ref ** 2).sum()) < TOL
            s.step(2)


def test_fp64_without_coulomb_is_the_free_motion():
    """No pair term and no bath: the trap alone, one ion at a time, to the last bit."""
    import paper_1907_10514_gb300 as it
    n = 70
    x = iongen.gaussian_positions(n, 30e-6, seed=5)
    p = it.make_params(None, precision=it.IONTRAP_PREC_FP64, Omega=iongen.OMEGA_RF, q=0.2, omega_z=2 * np.pi * 1e5,
                       dt=iongen.rf_period_dt(iongen.OMEGA_RF), flags=it.IONTRAP_COULOMB_OFF)
    with it.Simulation([iongen.CA40], np.zeros(n, np.uint8), x, None, p) as s:
        many = s.step(130).state()
    for i in (0, 31, 32, 69):
        with it.Simulation([iongen.CA40], np.zeros(1, np.uint8), x[:, i:i + 1], None, p) as s:
            one = s.step(130).state()
        assert np.array_equal(one[0][:, 0], many[0][:, i]) and np.array_equal(one[1][:, 0], many[1][:, i])
