"""Device memory of FP64 handles, and the forces and steps of those whose row blocks are summed in
several bands (above 16384 ions)."""
import numpy as np
import pytest

import iongen
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,megabytes", [(4096, 16), (16384, 64), (32768, 96), (131072, 300), (262144, 550), (1000000, 2100)])
def test_scratch_grows_with_n_not_its_square(n, megabytes):
    """Column slots of at most 64 row blocks of 256 ions (1536 bytes an ion), the state and the pair
    streams (137 bytes an ion), and per warp row and column slots (~10 MB)."""
    import paper_1907_10514_gb300 as it
    assert it.iontrap_estimate_bytes(n, it.IONTRAP_PREC_FP64) < megabytes * 1e6


def test_without_the_pair_term_there_are_no_slots():
    import paper_1907_10514_gb300 as it
    n = 200000
    x = iongen.gaussian_positions(n, 1e-3, seed=3)
    p = it.make_params(None, precision=it.IONTRAP_PREC_FP64, Omega=iongen.OMEGA_RF, q=0.2, omega_z=2 * np.pi * 1e5,
                       gamma=1e5, T_bath=1e-3, dt=iongen.rf_period_dt(iongen.OMEGA_RF), flags=it.IONTRAP_COULOMB_OFF)
    with it.Simulation([iongen.CA40], np.zeros(n, np.uint8), x, None, p) as s:
        assert it.iontrap_device_bytes(s.handle) < 220 * n
        many = s.step(3).state()
        assert not s.forces().any()
    with it.Simulation([iongen.CA40], np.zeros(2, np.uint8), x[:, :2], None, p) as s:  # the same noise: ions 0 and 1
        two = s.step(3).state()
    assert np.array_equal(two[0], many[0][:, :2]) and np.array_equal(two[1], many[1][:, :2])


# one band (64 row blocks of 256 ions), its last one ragged; two, the second of one ion; two full; three
@pytest.mark.parametrize("n", [16383, 16385, 32768, 33000])
@pytest.mark.parametrize("unit", [True, False])
def test_forces_and_steps_in_bands(n, unit):
    """The bound of the other FP64 force tests (terms within 3 ulp, sums of N terms): 1e-12."""
    import paper_1907_10514_gb300 as it
    rng = np.random.default_rng([n, 47])
    x = iongen.gaussian_positions(n, 30e-6 * (n / 512.0) ** (1 / 3), seed=[n, 19])
    sp = rng.integers(0, 3, n).astype(np.uint8)
    species = [iongen.Species(40.0, 1.0), iongen.Species(17.0, 1.0 if unit else 2.0),
               iongen.Species(137.0, 1.0 if unit else -1.0)]
    p = it.make_params(None, precision=it.IONTRAP_PREC_FP64, Omega=iongen.OMEGA_RF, q=0.2, omega_z=2 * np.pi * 1e5,
                       gamma=1e5, T_bath=1e-3, dt=iongen.rf_period_dt(iongen.OMEGA_RF), seed=3,
                       flags=it.IONTRAP_ALLOW_UNSTABLE)
    q, m, _ = oracle.ion_arrays(species, sp)
    idx = np.unique(np.r_[np.arange(40), rng.integers(0, n, 200), np.arange(n - 40, n), 16383 + np.arange(min(2, n - 16383))])
    with it.Simulation(species, sp, x, None, p) as s:
        for k in range(2):  # the initial positions, then those two steps on
            f = s.forces()
            ref = oracle.coulomb_accel(s.state()[0], q, m, idx=idx)
            assert np.sqrt(((f[:, idx] - ref) ** 2).sum() / (ref ** 2).sum()) < 1e-12
            s.step(2)
