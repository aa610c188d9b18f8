"""Dust temperatures where the tabulated inverse must not be used as it is: two
wavelengths whose emissions meet within a row of the table, with strengths for
which the last coefficient of the row's series vanishes (an emission per unit
mass of 2 to 2.125, the first row of an octave) although the series has not
ended."""
import numpy as np
import pytest

from paper_1410_1629_gb300 import rt
from paper_1410_1629_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU-only machines
    pytest.skip("no CUDA device", allow_module_level=True)


# strengths S kabs dlambda / lambda^5 at 0.125 and 8 um; the series of the row is
# off by 7e-11, 2e-11, 8e-10 and 1e-13 of T
@pytest.mark.parametrize("strength", [(1.267074356515321e18, 2.1695449970081087), (2.8158297872842244e19, 2.1695449970081087),
                                      (8.709781561950923e31, 4.772473184093586), (1.3017211267793224e16, 2.1695449970081087)])
def test_rows_whose_last_coefficient_vanishes(strength):
    from oracle import oracle as O
    rng = np.random.default_rng(6)
    # cells of width 1 and 1/2 (exact planes and masses), 2^16 of them: by the table
    grid = W.cartesian_grid([-32.0, 32.0, -32.0, 32.0, -4.0, 4.0], rng.lognormal(0.0, 1.0, (16, 64, 64)).astype(np.float32))
    wl = np.array([0.125, 8.0])
    edges = np.sqrt(wl[0] * wl[1]) * np.array([1.0 / 64.0, 1.0, 64.0])
    kappa = np.array(strength) * wl ** 5 / np.diff(edges)
    base = W.panchromatic_disk(n_cells=4, n_lambda=2, n_pix=8)
    prob = W.replace(base, grid=grid, wavelengths=wl, kappa=kappa, albedo=np.zeros(2), g=np.zeros(2),
                     sources=[W.replace(base.sources[0], lum=np.ones(2))])
    mass = grid.density.astype(np.float64).reshape(-1) * 0.5
    ab = np.zeros((2, grid.n_cells))
    ab[0] = mass * rng.uniform(1.8, 2.4, grid.n_cells)  # the row and its neighbours
    T_o, held_o = O.dust_temperature(prob, ab, 1.0)
    sim = rt.Simulation(prob)
    try:
        T_g, held_g = sim.dust_temperature(1.0, absorption=ab)
    finally:
        sim.close()
    # ln T carries 2 ulp of a number below 9.3 on both sides, E's rounding over its slope (at least 1) adds less
    np.testing.assert_allclose(T_g, T_o, rtol=1e-14, atol=0)
    assert held_g == held_o == 0


@pytest.mark.parametrize("shape", [(1, 127, 306), (1, 127, 307), (36, 36, 36)])  # 38862, 38989 (line: 38912) and 46656 cells
def test_grids_around_the_table_s_line(shape):
    from oracle import oracle as O
    rng = np.random.default_rng(8)
    nz, ny, nx = shape
    grid = W.cartesian_grid([0.0, float(nx), 0.0, float(ny), 0.0, float(nz)], rng.lognormal(0.0, 1.0, shape).astype(np.float32))
    n_lambda = 8
    wl = np.geomspace(0.1, 1000.0, n_lambda)
    kappa, albedo, g = W.panchromatic_optics(wl, 1.25)
    base = W.panchromatic_disk(n_cells=4, n_lambda=n_lambda, n_pix=8)
    prob = W.replace(base, grid=grid, wavelengths=wl, kappa=kappa, albedo=albedo, g=g,
                     sources=[W.replace(base.sources[0], lum=np.ones(n_lambda))])
    S = 1e11
    total = O.dust_emission(prob, np.exp(rng.uniform(np.log(0.7), np.log(1.4e4), grid.n_cells)), S).sum(axis=0)
    total[rng.uniform(size=total.size) < 0.05] = 0.0
    ab = np.full((n_lambda, 1), 1.0 / n_lambda) * total[None, :]
    T_o, held_o = O.dust_temperature(prob, ab, S)
    sim = rt.Simulation(prob)
    try:
        T_g, held_g = sim.dust_temperature(S, absorption=ab)
    finally:
        sim.close()
    np.testing.assert_allclose(T_g, T_o, rtol=1e-14, atol=0)  # (as above; exact planes and masses)
    assert held_g == held_o and held_o > 0
