"""The FP64 form's forces against an extended-precision sum."""
import numpy as np
import pytest

import iongen
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 33, 300])
@pytest.mark.parametrize("unit", [True, False])
def test_fp64_forces_to_the_last_digits(n, unit):
    """A term is within 3 ulp of its exact value, and the N additions of an ion's sum round by half
    an ulp of at most the sum of the terms' magnitudes each, in both directions: the error stays
    below (3 + sqrt N) 2^-52 of that sum."""
    import paper_1907_10514_gb300 as it
    rng = np.random.default_rng([n, 43])
    x = iongen.gaussian_positions(n, 30e-6, seed=[n, 17])
    sp = rng.integers(0, 2, n).astype(np.uint8)
    species = [iongen.Species(40.0, 1.0), iongen.Species(17.0, 1.0 if unit else 2.0)]
    p = it.make_params(None, precision=it.IONTRAP_PREC_FP64, Omega=iongen.OMEGA_RF, q=0.2, omega_z=2 * np.pi * 1e5,
                       dt=iongen.rf_period_dt(iongen.OMEGA_RF), flags=it.IONTRAP_ALLOW_UNSTABLE)
    with it.Simulation(species, sp, x, None, p) as s:
        f = s.forces()
    L = np.longdouble
    z, M = np.array([s.charge_e for s in species])[sp], np.array([s.mass_amu for s in species])[sp]
    w = L(oracle.const("e")) ** 2 / (4 * L(np.pi) * L(oracle.const("eps0"))) * z.astype(L)[:, None] * z.astype(L)[None, :]
    d = x.astype(L)[:, :, None] - x.astype(L)[:, None, :]
    r2 = (d * d).sum(axis=0)
    np.fill_diagonal(r2, L(1))
    t = w * d / (r2 * np.sqrt(r2)) / (M * oracle.const("amu")).astype(L)[:, None]
    # the library's factor k_e e^2 z / M is a double of a few roundings: one common factor per species
    ref, mag = t.sum(axis=2), np.abs(t).sum(axis=2)
    for k in range(2):
        on = sp == k
        if not on.any():
            continue
        g = (f[:, on] * ref[:, on]).sum() / (ref[:, on] ** 2).sum()
        assert abs(g - 1) < 1e-14
        assert (np.abs(f[:, on] / g - ref[:, on]) / mag[:, on]).max() < (3 + np.sqrt(n)) * 2.0 ** -52
