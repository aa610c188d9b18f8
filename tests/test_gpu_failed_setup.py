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
