"""The sorted pass's order of the cells is made when a grid gets its first
instrument: launches with and without it agree, a grid without instruments runs,
and a grid that replaces another in the same context gets its own order."""
import numpy as np
import pytest

from paper_1410_1629_gb300 import rt
from paper_1410_1629_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU-only machines
    pytest.skip("no CUDA device", allow_module_level=True)

import parity as PAR  # noqa: E402


def _tree(kind, seed):
    make = W.clumpy_octree if kind == "octree" else W.clumpy_bintree
    return make(n_particles=1000 + 500 * seed, n_samples=30_000, target_leaves=1500 + 700 * seed, max_level=6, n_lambda=2,
                n_pix=16)


def _same(a, b):
    assert np.array_equal(a["counters"], b["counters"]) and a["raw_stats"]["device_flags"] == 0
    bound = 2.0 * a["raw_stats"]["peeloffs"] * 2.0 ** -53
    for x, y in zip(a["images"], b["images"]):
        np.testing.assert_allclose(x, y, rtol=bound, atol=0)


def test_grids_replaced_in_one_context():
    probs = [_tree("octree", 0), W.voronoi_disk(n_sites=700, n_lambda=2, n_pix=16), _tree("bintree", 1), _tree("octree", 2),
             _tree("octree", 0)]
    n = 1500
    refs = [PAR.gpu_run(p, n, inline_peels=1) for p in probs]
    sim = rt.Simulation(probs[0])
    try:
        for k, p in enumerate(probs):
            if k:
                desc, keep = rt.grid_desc(p.grid)
                rt.rt_create_grid(sim.ctx, desc)
                del keep
                rt.rt_set_optics(sim.ctx, 0, p.kappa, p.albedo, p.g, p.wavelengths)
                rt.rt_add_sources(sim.ctx, [rt.source_desc(s) for s in p.sources], [s.lum for s in p.sources])
                rt.rt_add_instruments(sim.ctx, [rt.instrument_desc(q) for q in p.instruments])
                sim.problem, sim.n_lambda, sim.n_cells = p, p.n_lambda, p.grid.n_cells
            if k % 2:  # a launch in place first on some of them
                _same(PAR.gpu_run(p, n, sim=sim, inline_peels=1), refs[k])
                sim.reset()
            for _ in range(2):
                got = PAR.gpu_run(p, n, sim=sim)
                assert got["raw_stats"]["sorted_peels"] > 0
                _same(got, refs[k])
                sim.reset()
    finally:
        sim.close()


def test_instruments_added_after_launches():
    """Launches without instruments, then the frames one by one."""
    p = _tree("bintree", 1)
    ref = PAR.gpu_run(p, 1500, inline_peels=1)
    sim = rt.Simulation(W.replace(p, instruments=[]))
    try:
        sim.launch(1500, 0, 0)
        np.testing.assert_allclose(sim.absorption().cpu().numpy(), ref["absorption"],
                                   rtol=2.0 * ref["raw_stats"]["path_crossings"] * 2.0 ** -53, atol=0)
        for q in p.instruments:
            rt.rt_add_instruments(sim.ctx, [rt.instrument_desc(q)])
        sim.problem = p
        sim.reset()
        got = PAR.gpu_run(p, 1500, sim=sim)
        assert got["raw_stats"]["sorted_peels"] > 0
        _same(got, ref)
    finally:
        sim.close()
