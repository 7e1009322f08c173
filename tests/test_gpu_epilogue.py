"""The separate epilogue (form 0), launched ahead of the pair sums or after them, gives the bits of
the merge by the last CTA of an i-block (form 1) over the same j-ranges."""
import numpy as np
import pytest

import iongen

pytestmark = pytest.mark.gpu


def _handle(it, n, charges, laser, flags):
    rng = np.random.default_rng([n, 23])
    x = iongen.gaussian_positions(n, 60e-6, seed=[n, 7])
    v = rng.normal(size=(3, n))
    sp = (np.arange(n) % 3 == 2).astype(np.uint8)
    species = [iongen.Species(iongen.CA40_AMU, charges[0]), iongen.Species(iongen.NH3_AMU, charges[1])]
    p = it.make_params(None, Omega=iongen.OMEGA_RF, q=0.2, omega_z=2 * np.pi * 0.1e6, gamma=1e5, T_bath=1e-3,
                       dt=iongen.rf_period_dt(iongen.OMEGA_RF), seed=n, flags=flags | it.IONTRAP_ALLOW_UNSTABLE)
    s = it.Simulation(species, sp, x, v, p)
    if laser:
        s.set_params(p, [(1e5, 1e-3, (3e5, -2e5, 1e5)), (0.0, 0.0, (0.0, 1e5, 0.0))])
    return s


# the edges of an epilogue CTA (64 ions) and of its groups of splits (8): 1 to 64 splits of one to
# several chunks; the default above 8192 ions
@pytest.mark.parametrize("n,T,I,packed,jsplit", [
    (1, 64, 2, 1, 1), (63, 64, 2, 1, 8), (64, 64, 2, 1, 8), (65, 64, 2, 1, 8), (129, 64, 1, 0, 129),
    (700, 64, 2, 1, 11), (1000, 128, 4, 1, 300), (8193, 64, 2, 1, 320),
])
@pytest.mark.parametrize("charges,laser,flag", [((1.0, 1.0), True, ""), ((1.0, 2.0), False, ""),
                                                ((1.0, 1.0), False, "IONTRAP_COULOMB_OFF")])
def test_separate_epilogue_gives_the_bits_of_the_last_cta(n, T, I, packed, jsplit, charges, laser, flag):
    import paper_1907_10514_gb300 as it
    got = []
    for fused, pdl, graph in ((1, 0, 0), (0, 0, 0), (0, 1, 0), (0, 1, 1)):
        with _handle(it, n, charges, laser, getattr(it, flag) if flag else 0) as s:
            s.set_config(T, I, packed, jsplit, fused, pdl, graph)
            s.step(45)
            x, v, a, step = s.checkpoint()
            assert step == 45
            s.restore(x, v, np.zeros_like(a), step)
            f = s.forces()
            s.step(3)
            got.append((x, v, a, f, *s.state()[:2]))
    for other in got[1:]:
        for u, w in zip(got[0], other):
            assert np.isfinite(u).all() and np.array_equal(u, w)
