"""Dust temperatures from the tabulated inverse of the emission (grids of 2^16
cells and more) against the oracle's bisection, over the whole range of
temperatures and on wavelength grids whose emission underflows at the cold
end."""
import numpy as np
import pytest

from paper_1410_1629_gb300 import rt
from paper_1410_1629_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU-only machines
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("nz", [8, 16])  # 32768 cells: solved one by one; 65536: by the table
@pytest.mark.parametrize("lo,hi,n_lambda", [(0.1, 1000.0, 24), (0.1, 1.0, 9), (5.0, 5000.0, 2)])
def test_temperatures_over_the_whole_range(nz, lo, hi, n_lambda):
    from oracle import oracle as O
    rng = np.random.default_rng(5)
    base = W.panchromatic_disk(n_cells=4, n_lambda=n_lambda, n_pix=8)
    # cells of width 1 and 1/2: their planes, and so their masses, are exact
    # (the planes' rounding would enter T by up to 1e-14 where E is linear in T)
    grid = W.cartesian_grid([-32.0, 32.0, -32.0, 32.0, -4.0, 4.0],
                            rng.lognormal(0.0, 1.0, (nz, 64, 64)).astype(np.float32))
    wl = np.geomspace(lo, hi, n_lambda)
    kappa, albedo, g = W.panchromatic_optics(wl, 1.25)
    prob = W.replace(base, grid=grid, wavelengths=wl, kappa=kappa, albedo=albedo, g=g,
                     sources=[W.replace(base.sources[0], lum=np.ones(n_lambda))])
    S = 1e11
    T0 = np.exp(rng.uniform(np.log(0.7), np.log(1.4e4), prob.grid.n_cells))  # beyond both limits
    total = O.dust_emission(prob, T0, S).sum(axis=0)
    total[rng.uniform(size=total.size) < 0.05] = 0.0
    share = rng.uniform(0.1, 1.0, n_lambda)
    ab = (share / share.sum())[:, None] * total[None, :]
    T_o, held_o = O.dust_temperature(prob, ab, S)
    sim = rt.Simulation(prob)
    try:
        T_g, held_g = sim.dust_temperature(S, absorption=ab)
        # ln T carries 2 ulp of a number below 9.3 on both sides, E's rounding
        # over its slope adds less
        np.testing.assert_allclose(T_g, T_o, rtol=1e-14, atol=0)
        assert held_g == held_o and held_o > 0
    finally:
        sim.close()
