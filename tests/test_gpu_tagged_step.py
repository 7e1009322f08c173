"""The tagged launch of row-persistent simulations gives the bits of the grid launch of the same
shape.  Launches with a wait limit of their own (iontrap_test_stall) take the grid's counter."""
import numpy as np
import pytest

import iongen

pytestmark = pytest.mark.gpu


def _handle(it, n, charges, laser, flags):
    rng = np.random.default_rng([n, 19])
    x = iongen.gaussian_positions(n, 40e-6, seed=[n, 5])
    v = rng.normal(size=(3, n))
    sp = (np.arange(n) % 3 == 2).astype(np.uint8)
    species = [iongen.Species(iongen.CA40_AMU, charges[0]), iongen.Species(iongen.NH3_AMU, charges[1])]
    p = it.make_params(None, Omega=iongen.OMEGA_RF, q=0.2, omega_z=2 * np.pi * 0.1e6, gamma=1e5, T_bath=1e-3,
                       dt=iongen.rf_period_dt(iongen.OMEGA_RF), seed=n, flags=flags | it.IONTRAP_ALLOW_UNSTABLE)
    s = it.Simulation(species, sp, x, v, p)
    if laser:
        s.set_params(p, [(1e5, 1e-3, (3e5, -2e5, 1e5)), (0.0, 0.0, (0.0, 1e5, 0.0))])
    return s


# (n, ions per thread, ions per CTA): the edges of the range (168 | 169, 2047, 2128 at parts of
# a chunk), 8, 16 and 24 reads in flight, one owner warp and four, a last CTA of one ion, parts
# without ions, odd counts; shapes next to those taken (43 ions per CTA, parts above a chunk)
@pytest.mark.parametrize("n,ipt,R", [
    (2, 1, 1), (150, 2, 42), (168, 1, 2), (169, 1, 2), (321, 1, 3), (433, 2, 32), (500, 1, 43), (600, 1, 42),
    (911, 1, 7), (1000, 1, 10), (1057, 2, 8), (1500, 1, 10), (2047, 1, 14), (2127, 1, 14), (2100, 1, 15),
])
@pytest.mark.parametrize("charges,laser,pseudo", [((1.0, 1.0), True, False), ((1.0, 2.0), False, False),
                                                  ((1.0, 1.0), False, True)])
def test_tagged_steps_are_the_grid_steps_bit_for_bit(n, ipt, R, charges, laser, pseudo):
    import paper_1907_10514_gb300 as it
    got = []
    for grid in (False, True):
        with _handle(it, n, charges, laser, it.IONTRAP_PSEUDO if pseudo else 0) as s:
            s.set_config(256, ipt, 1, R, 5, 0, 0)
            if grid:
                it.iontrap_test_stall(s.handle, 2_000_000_000, -1, 0)
            for k in (1, 2, 45):
                s.step(k)
            x, v, a, step = s.checkpoint()
            assert step == 48
            s.restore(x, v, a, step - 2)  # step indices repeat: tags must not
            s.step(3)
            got.append((x, v, a, s.state()[0]))
    for u, w in zip(*got):
        assert np.isfinite(u).all() and np.array_equal(u, w)
