"""Launches recorded into a CUDA graph on grids whose frames partly look along
an axis: the peel-offs that walk do so in place, replays add up, and plain
launches before and after them take the sorted pass."""
import numpy as np
import pytest

from paper_1410_1629_gb300 import rt
from paper_1410_1629_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU-only machines
    pytest.skip("no CUDA device", allow_module_level=True)

import parity as PAR  # noqa: E402


@pytest.mark.parametrize("walk_peels", [0, 1])
def test_cartesian_launch_captured_into_a_graph(walk_peels):
    """Three replays equal three plain launches up to the order of the FP64
    additions (2 n 2^-53 for n of them); a plain launch whose count is still
    outstanding when the capture begins, and plain launches afterwards, work."""
    prob = W.disk_galaxy(n_cells=24, n_lambda=2, n_pix=24, channels=3)
    n = 700
    ref = PAR.gpu_run(prob, n, walk_peels=walk_peels)
    assert ref["raw_stats"]["sorted_peels"] > 0
    sim = rt.Simulation(prob)
    try:
        sim.launch(n, walk_peels=walk_peels)
        sim.reset()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            sim.launch(n, 0, None, stream=torch.cuda.current_stream().cuda_stream, walk_peels=walk_peels)
        for _ in range(3):
            graph.replay()
        torch.cuda.synchronize()
        st = sim.stats()
        assert st["device_flags"] == 0 and st["sorted_peels"] == 0
        for k in ("crossings", "events", "peeloffs", "packets", "column_peels"):
            assert st[k] == 3 * ref["raw_stats"][k]
        bound = 2.0 * st["peeloffs"] * 2.0 ** -53
        for x, y in zip(sim.images(), ref["images"]):
            np.testing.assert_allclose(x.cpu().numpy(), 3.0 * y, rtol=bound, atol=0)
        for _ in range(2):
            sim.reset()
            again = PAR.gpu_run(prob, n, sim=sim, walk_peels=walk_peels)
            assert again["raw_stats"]["sorted_peels"] == ref["raw_stats"]["sorted_peels"]
            for x, y in zip(again["images"], ref["images"]):
                np.testing.assert_allclose(x, y, rtol=bound, atol=0)
    finally:
        sim.close()
