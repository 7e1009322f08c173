"""The bounded waits of the kernels that default handles step on, made to expire without a fault:
one CTA keeps its positions to itself (iontrap_test_stall) under a limit of 1 ms.  Every warp of
every CTA then leaves the launch at one step; the status is IONTRAP_ETIMEOUT, the state is the one
the launch started from, and the next handle steps as if nothing had been."""
import time

import numpy as np
import pytest

import iongen

pytestmark = pytest.mark.gpu

LIMIT_NS = 1_000_000  # 1 ms: a step of these clouds takes 1 to 5 us
K = 60                # steps of the launch


def _handle(it, n, laser):
    rng = np.random.default_rng([n, 31])
    x = iongen.gaussian_positions(n, 30e-6, seed=[n, 11])
    v = rng.normal(size=(3, n))
    sp = (np.arange(n) % 3 == 2).astype(np.uint8)
    p = it.make_params(None, Omega=iongen.OMEGA_RF, q=0.2, omega_z=2 * np.pi * 0.1e6, gamma=1e5, T_bath=1e-3,
                       dt=iongen.rf_period_dt(iongen.OMEGA_RF), seed=n, flags=it.IONTRAP_ALLOW_UNSTABLE)
    s = it.Simulation([iongen.CA40, iongen.NH3], sp, x, v, p)
    if laser:
        s.set_params(p, [(1e5, 1e-3, (3e5, -2e5, 1e5)), (0.0, 0.0, (0.0, 1e5, 0.0))])
    return s


# default handles: clusters of 4, 8 and 16 CTAs; tagged positions with 8, 16 and 24 reads in flight
# and a last CTA of fewer ions
CASES = [(13, "CLUSTER", 4), (64, "CLUSTER", 8), (150, "CLUSTER", 16),
         (300, "TAGGED", 150), (1000, "TAGGED", 143), (2047, "TAGGED", 147)]


@pytest.mark.parametrize("n,kernel,ctas", CASES)
@pytest.mark.parametrize("laser", [False, True])
@pytest.mark.parametrize("cta,at", [(0, 0), (-1, 5), (1, 6), (-1, K - 2)])
def test_a_withheld_step_ends_the_launch(n, kernel, ctas, laser, cta, at):
    import paper_1907_10514_gb300 as it
    cta %= ctas
    with _handle(it, n, laser) as s:
        x0, v0, a0, _ = s.checkpoint()
        for bad in (ctas, ctas + 1):  # no such CTA
            with pytest.raises(it.IonTrapError) as e:
                it.iontrap_test_stall(s.handle, LIMIT_NS, bad, 0)
            assert e.value.code == it.IONTRAP_EINVAL
        it.iontrap_test_stall(s.handle, LIMIT_NS, cta, at)
        assert it.iontrap_test_step_kernel(s.handle) == (getattr(it, "IONTRAP_KERNEL_" + kernel), ctas)
        t0 = time.perf_counter()
        s.step(K)
        with pytest.raises(it.IonTrapError) as e:
            s.sync()
        assert e.value.code == it.IONTRAP_ETIMEOUT
        assert time.perf_counter() - t0 < 1.0  # the limit, not the default 2 s
        x, v, step, _ = it.iontrap_state(s.handle, n, accept=(it.IONTRAP_ETIMEOUT,))
        assert step == 0
        assert np.array_equal(x, x0) and np.array_equal(v, v0)
        with pytest.raises(it.IonTrapError) as e:  # sticky
            s.step(1)
        assert e.value.code == it.IONTRAP_ETIMEOUT


@pytest.mark.parametrize("n,kernel,ctas", CASES)
def test_a_limit_that_is_not_reached_changes_nothing(n, kernel, ctas):
    import paper_1907_10514_gb300 as it
    got = []
    for limit in (False, True):
        with _handle(it, n, True) as s:
            if limit:  # the stall lies beyond every launch
                it.iontrap_test_stall(s.handle, 200_000_000, 0, 1 << 40)
            assert it.iontrap_test_step_kernel(s.handle) == (getattr(it, "IONTRAP_KERNEL_" + kernel), ctas)
            for k in (1, 2, K):
                s.step(k)
            got.append(s.checkpoint())
    for u, w in zip(*got):
        assert np.array_equal(u, w)


def test_a_withheld_last_arrival_is_a_timeout_too():
    """The grid counts its CTAs once after a launch's last step."""
    import paper_1907_10514_gb300 as it
    n = 300
    with _handle(it, n, False) as s:
        it.iontrap_test_stall(s.handle, LIMIT_NS, 7, K - 1)
        assert it.iontrap_test_step_kernel(s.handle)[0] == it.IONTRAP_KERNEL_TAGGED
        s.step(K)
        with pytest.raises(it.IonTrapError) as e:
            s.sync()
        assert e.value.code == it.IONTRAP_ETIMEOUT
        x, v, step, _ = it.iontrap_state(s.handle, n, accept=(it.IONTRAP_ETIMEOUT,))
        assert step == 0


@pytest.mark.parametrize("cta,barrier", [(0, 0), (3, 7), (-1, 2)])
def test_a_withheld_barrier_ends_a_minimisation(cta, barrier):
    """The iterations' barriers on the grid (above 432 ions)."""
    import paper_1907_10514_gb300 as it
    n = 1030
    x = iongen.gaussian_positions(n, 30e-6, seed=[n, 29])
    p = it.make_params(None, Omega=iongen.OMEGA_RF, q=0.2, omega_z=2 * np.pi * 1e5, dt=iongen.rf_period_dt(iongen.OMEGA_RF),
                       flags=it.IONTRAP_PSEUDO)
    want = None
    for stall in (False, True):
        with it.Simulation([iongen.CA40], np.zeros(n, np.uint8), x, None, p) as s:
            ctas = it.iontrap_test_step_kernel(s.handle)[1]
            if not stall:  # beyond every launch: the limit alone changes nothing
                it.iontrap_test_stall(s.handle, 200_000_000, cta % ctas, 1 << 40)
                want = s.minimize(20, 5e-7, 0.0, 5e-8)
                assert want[0] == 20
                continue
            it.iontrap_test_stall(s.handle, LIMIT_NS, cta % ctas, barrier)
            t0 = time.perf_counter()
            with pytest.raises(it.IonTrapError) as e:
                s.minimize(20, 5e-7, 0.0, 5e-8)
            assert e.value.code == it.IONTRAP_ETIMEOUT and time.perf_counter() - t0 < 1.0
            with pytest.raises(it.IonTrapError) as e:  # sticky
                s.minimize(20, 5e-7, 0.0, 5e-8)
            assert e.value.code == it.IONTRAP_ETIMEOUT
    with it.Simulation([iongen.CA40], np.zeros(n, np.uint8), x, None, p) as s:
        assert s.minimize(20, 5e-7, 0.0, 5e-8) == want
