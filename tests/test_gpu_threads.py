"""Contexts in several threads: octrees of different depth, whose kernels need
different amounts of shared memory, launched side by side."""
import threading

import numpy as np
import pytest

from paper_1410_1629_gb300 import rt
from paper_1410_1629_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU-only machines
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("inline_peels", [0, 1])
def test_octrees_of_different_depth_in_two_threads(inline_peels):
    rounds, n = 2000, 4
    sims = [rt.Simulation(W.clumpy_octree(n_particles=500, n_samples=5000, target_leaves=300, max_level=level, n_lambda=1,
                                          n_pix=8)) for level in (3, 9)]
    failed = [[], []]

    def go(i):
        stream = torch.cuda.Stream().cuda_stream
        for _ in range(rounds):
            try:
                sims[i].launch(n, 0, 1, stream=stream, inline_peels=inline_peels)
            except rt.RTError as e:
                failed[i].append(str(e))

    try:
        threads = [threading.Thread(target=go, args=(i,)) for i in range(2)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        torch.cuda.synchronize()
        assert failed == [[], []]
        for s in sims:
            st = s.stats()
            assert st["device_flags"] == 0 and st["packets"] == rounds * n
            images = [t.cpu().numpy() for t in s.images()]
            s.reset()
            s.launch(n, 0, 1, inline_peels=1)
            one = s.stats()
            assert st["crossings"] == rounds * one["crossings"] and st["peeloffs"] == rounds * one["peeloffs"]
            for x, y in zip(images, s.images()):
                np.testing.assert_allclose(x, rounds * y.cpu().numpy(), rtol=2.0 * st["peeloffs"] * 2.0 ** -53, atol=0)
    finally:
        for s in sims:
            s.close()
