"""The mass-weighted Hessian against an extended-precision evaluation."""
import numpy as np
import pytest

import iongen
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [131, 300])
@pytest.mark.parametrize("charges", [(1.0, 1.0), (1.0, 2.0)])
def test_hessian_blocks_to_the_last_digits(n, charges):
    """An entry comes of ten roundings (a difference, y^3, y^5, the series, charge, two factors of r,
    weight and its product), each of at most 2^-53 and uniform: 2.0e-16 rms.  The divisions and the
    root of the textbook form, or a rounded r^2, make 2.5e-16 to 2.7e-16.  Mean over the
    off-diagonal blocks of the largest error over the largest entry: below 2.3e-16; a block's worst
    is below fifteen half ulps.  The factor k_e e^2 z z' / sqrt(M M') of a pair of species is a double
    of a few roundings, common to its blocks, and taken out."""
    import paper_1907_10514_gb300 as it
    x = iongen.gaussian_positions(n, 30e-6, seed=[n, 53])
    sp = (np.arange(n) % 5 == 4).astype(np.uint8)
    species = [iongen.Species(iongen.CA40_AMU, charges[0]), iongen.Species(iongen.NH3_AMU, charges[1])]
    p = it.make_params(None, Omega=iongen.OMEGA_RF, q=0.2, omega_z=2 * np.pi * 1e5, dt=iongen.rf_period_dt(iongen.OMEGA_RF),
                       flags=it.IONTRAP_PSEUDO | it.IONTRAP_ALLOW_UNSTABLE)
    with it.Simulation(species, sp, x, None, p) as s:
        H = s.hessian().reshape(n, 3, n, 3)
    L = np.longdouble
    z, M = np.array(charges, L)[sp], np.array([s.mass_amu * oracle.const("amu") for s in species])[sp].astype(L)
    ke2 = L(1.0 / (4.0 * np.pi * oracle.const("eps0")) * oracle.const("e") * oracle.const("e"))
    d = x.astype(L)[:, :, None] - x.astype(L)[:, None, :]
    r2 = (d * d).sum(axis=0)
    np.fill_diagonal(r2, L(1))
    k3 = ke2 * z[:, None] * z[None, :] / (r2 * np.sqrt(r2)) / np.sqrt(M[:, None] * M[None, :])
    ref = np.stack([[k3 * ((1 if a == b else 0) - 3 * d[a] * d[b] / r2) for b in range(3)] for a in range(3)])
    got = H.transpose(1, 3, 0, 2).astype(L)
    along = (got * ref).sum(axis=(0, 1)) / (ref * ref).sum(axis=(0, 1))
    for s in range(2):
        for t in range(2):
            on = (sp[:, None] == s) & (sp[None, :] == t) & ~np.eye(n, dtype=bool)
            g = along[on].mean()
            assert abs(g - 1) < 1e-15
            rel = (np.abs(got / g - ref).max(axis=(0, 1)) / np.abs(ref).max(axis=(0, 1)))[on].astype(float)
            assert rel.mean() < 2.3e-16 and rel.max() < 15 * 2.0 ** -53
