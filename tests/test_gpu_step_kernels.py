"""The cluster and the tagged launch of row-persistent steps give the bits of the grid launch with
its counter: on shapes that take each of them, with the kernel that steps asserted on both sides."""
import numpy as np
import pytest

import iongen

pytestmark = pytest.mark.gpu


def _handle(it, n, charges, laser, flags):
    rng = np.random.default_rng([n, 37])
    x = iongen.gaussian_positions(n, 40e-6, seed=[n, 13])
    v = rng.normal(size=(3, n))
    sp = (np.arange(n) % 3 == 2).astype(np.uint8)
    species = [iongen.Species(iongen.CA40_AMU, charges[0]), iongen.Species(iongen.NH3_AMU, charges[1])]
    p = it.make_params(None, Omega=iongen.OMEGA_RF, q=0.2, omega_z=2 * np.pi * 0.1e6, gamma=1e5, T_bath=1e-3,
                       dt=iongen.rf_period_dt(iongen.OMEGA_RF), seed=n, flags=flags | it.IONTRAP_ALLOW_UNSTABLE)
    s = it.Simulation(species, sp, x, v, p)
    if laser:
        s.set_params(p, [(1e5, 1e-3, (3e5, -2e5, 1e5)), (0.0, 0.0, (0.0, 1e5, 0.0))])
    return s


# (n, threads, ions per thread, ions per CTA): clusters of 1, 4, 8 and 16 at their edges, up to 432
# in shapes of 512 threads (those of 256 are tagged above 168 ions); tagged launches with 8, 16 and
# 24 reads in flight for one and two ions per thread; shapes that neither takes
@pytest.mark.parametrize("kernel,n,threads,ipt,R", [
    ("CLUSTER", 12, 512, 1, 4), ("CLUSTER", 13, 256, 1, 3), ("CLUSTER", 28, 256, 2, 9), ("CLUSTER", 29, 256, 1, 7),
    ("CLUSTER", 84, 512, 2, 40), ("CLUSTER", 85, 256, 1, 1), ("CLUSTER", 168, 256, 1, 2), ("CLUSTER", 169, 512, 1, 2),
    ("CLUSTER", 321, 512, 1, 3), ("CLUSTER", 431, 512, 1, 32), ("CLUSTER", 432, 512, 2, 30),
    ("TAGGED", 169, 256, 1, 2), ("TAGGED", 321, 256, 1, 3), ("TAGGED", 433, 256, 2, 32), ("TAGGED", 1000, 256, 1, 10),
    ("TAGGED", 1057, 256, 2, 8), ("TAGGED", 2047, 256, 1, 14), ("TAGGED", 2100, 256, 2, 28),
    ("GRID", 433, 512, 1, 3), ("GRID", 500, 256, 1, 43),
])
@pytest.mark.parametrize("charges,laser,pseudo", [((1.0, 1.0), True, False), ((1.0, 2.0), False, False),
                                                  ((1.0, 1.0), False, True)])
def test_steps_are_the_grid_steps_bit_for_bit(kernel, n, threads, ipt, R, charges, laser, pseudo):
    import paper_1907_10514_gb300 as it
    got = []
    for grid in (False, True):
        with _handle(it, n, charges, laser, it.IONTRAP_PSEUDO if pseudo else 0) as s:
            s.set_config(threads, ipt, 1, R, 5, 0, 0)
            if grid:  # a limit without a stall
                it.iontrap_test_stall(s.handle, 2_000_000_000, -1, 0)
            want = it.IONTRAP_KERNEL_GRID if grid else getattr(it, "IONTRAP_KERNEL_" + kernel)
            assert it.iontrap_test_step_kernel(s.handle)[0] == want
            for k in (1, 2, 45):
                s.step(k)
            x, v, a, step = s.checkpoint()
            assert step == 48
            s.restore(x, v, a, step - 2)  # step indices repeat: tags must not
            s.step(3)
            got.append((x, v, a, s.state()[0]))
    for u, w in zip(*got):
        assert np.isfinite(u).all() and np.array_equal(u, w)
