"""The allocation-free force kernel at the edges of its j-ranges, chunks and ion blocks: bit
for bit the forces of a handle in the last-CTA form over the same j-ranges."""
import numpy as np
import pytest

import iongen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 33, 64, 127, 128, 129, 300, 513, 700, 896, 1025, 2800, 2801, 3200, 3201, 4099, 6144, 6145, 7169, 8191, 8192])
@pytest.mark.parametrize("unit", [True, False])
def test_noalloc_forces_are_the_last_cta_forces(n, unit):
    import torch
    import paper_1907_10514_gb300 as it
    rng = np.random.default_rng([n, 31])
    species = [iongen.CA40, iongen.Species(17.0, 1.0 if unit else -2.0)]
    sp = rng.integers(0, 2, n).astype(np.uint8)
    x = iongen.gaussian_positions(n, 40e-6, seed=[n, 5])
    x[:, 0] = 0.0  # a coordinate whose split takes the plain conversions
    x[1, n // 2] = 1e-40
    p = it.make_params(None, Omega=iongen.OMEGA_RF, dt=1e-8, flags=it.IONTRAP_TRAP_OFF)
    splits = min(8, max(1, -(-n // 128)))
    with it.Simulation(species, sp, x, None, p) as s:
        s.set_config(64, 1, 0, -(-n // splits), 1)
        want = s.forces()
    d_x, d_sp = torch.from_numpy(x).cuda(), torch.from_numpy(sp).cuda()
    out = [torch.full((3, n), float("nan"), dtype=torch.float64, device="cuda") for _ in range(2)]
    streams = [torch.cuda.Stream() for _ in out]
    torch.cuda.synchronize()
    for o, st in zip(out, streams):  # overlapping calls do not share anything
        it.iontrap_forces_noalloc(species, d_sp.data_ptr(), d_x.data_ptr(), n, o.data_ptr(), st)
    torch.cuda.synchronize()
    for o in out:
        assert np.array_equal(o.cpu().numpy(), want)
