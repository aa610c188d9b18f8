"""Set-up calls that run out of device memory leave a context that works."""
import numpy as np
import pytest

from paper_1410_1629_gb300 import rt
from paper_1410_1629_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU-only machines
    pytest.skip("no CUDA device", allow_module_level=True)


def test_launch_after_a_failed_allocation():
    """The failed call's CUDA error is not found again by the next launch's check."""
    prob = W.uniform_cube(n_cells=4, n_pix=16, channels=3)
    wl = np.geomspace(0.1, 1000.0, 64)
    prob = W.replace(prob, wavelengths=wl, kappa=np.ones(64), albedo=np.full(64, 0.5), g=np.zeros(64),
                     sources=[W.replace(prob.sources[0], lum=np.ones(64))])
    sim = rt.Simulation(prob)
    try:
        sim.launch(100, 0, 3)
        st_ref = sim.stats()
        q = rt.instrument_desc(prob.instruments[0])
        q.nx = q.ny = 1 << 14  # 412 GB of images
        with pytest.raises(rt.RTError) as err:
            rt.rt_add_instruments(sim.ctx, [q])
        assert err.value.status == rt.RT_ERR_OOM
        sim.reset()
        sim.launch(100, 0, 3)
        st = sim.stats()
        assert st["device_flags"] == 0 and st["crossings"] == st_ref["crossings"]
    finally:
        sim.close()


def _set_up(ctx, prob, layout):
    desc, keep = rt.grid_desc(prob.grid)
    desc.layout = layout
    rt.rt_create_grid(ctx, desc)
    del keep
    rt.rt_set_optics(ctx, 0, prob.kappa, prob.albedo, prob.g, prob.wavelengths)
    rt.rt_add_sources(ctx, [rt.source_desc(s) for s in prob.sources], [s.lum for s in prob.sources])
    rt.rt_add_instruments(ctx, [rt.instrument_desc(q) for q in prob.instruments])


def test_grid_creation_out_of_memory():
    """A grid creation that fails half-way: the buffers it had got come back with
    their own sizes."""
    base = W.uniform_cube(n_cells=4, n_pix=16)
    rng = np.random.default_rng(1)
    # 134 MB of densities in one buffer (row-major), and 84 MB in two (stored z fastest)
    big = W.replace(base, grid=W.cartesian_grid([-1, 1] * 3, rng.uniform(0.1, 1.0, (256, 256, 512)).astype(np.float32)))
    other = W.replace(base, grid=W.cartesian_grid([-1, 1] * 3, np.ones((320, 256, 256), np.float32)))
    n = 2000
    sim = rt.Simulation(big, layout=rt.RT_LAYOUT_ROW_MAJOR)
    hold = None
    try:
        sim.launch(n, 0, 3)
        ref, st_ref = sim.images()[0].cpu().numpy(), sim.stats()
        # a new context that holds nothing but the densities
        rt.rt_context_destroy(sim.ctx)
        sim.ctx = rt.rt_context_create(0)
        desc, keep = rt.grid_desc(big.grid)
        desc.layout = rt.RT_LAYOUT_ROW_MAJOR
        rt.rt_create_grid(sim.ctx, desc)
        del keep
        free = torch.cuda.mem_get_info()[0]
        hold = torch.empty(free - (24 << 20), dtype=torch.uint8, device="cuda")
        with pytest.raises(rt.RTError) as err:  # its first buffer fits in place of the old density, its second does not
            desc, keep = rt.grid_desc(other.grid)
            rt.rt_create_grid(sim.ctx, desc)
        assert err.value.status == rt.RT_ERR_OOM
        del hold
        hold = None
        torch.cuda.empty_cache()
        for _ in range(2):  # the same context again: its buffers new, then from the pool
            _set_up(sim.ctx, big, rt.RT_LAYOUT_ROW_MAJOR)
            sim.launch(n, 0, 3)
            st = sim.stats()
            assert st["device_flags"] == 0 and st["crossings"] == st_ref["crossings"]
            np.testing.assert_allclose(sim.images()[0].cpu().numpy(), ref, rtol=2.0 * st["peeloffs"] * 2.0 ** -53, atol=0)
    finally:
        del hold
        torch.cuda.empty_cache()
        sim.close()
