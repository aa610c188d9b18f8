"""The routes a launch can take give the same results: peel-offs in the sorted
pass or walked in place on every grid, instruments that share a view's walks
or not, launches around the sizes where the packet slots fill, and batches
around the run lengths.  Two routes add the same positive FP64 contributions in
different orders, so a sum of n of them differs by at most 2 n 2^-53 relative."""
import dataclasses

import numpy as np
import pytest

from paper_1410_1629_gb300 import rt
from paper_1410_1629_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU-only machines
    pytest.skip("no CUDA device", allow_module_level=True)

import parity as PAR  # noqa: E402


def _order_bound(n_terms):
    return 2.0 * float(n_terms) * 2.0 ** -53


def _assert_same(a, b):
    assert np.array_equal(a["counters"], b["counters"])
    assert a["raw_stats"]["device_flags"] == b["raw_stats"]["device_flags"] == 0
    st = a["raw_stats"]
    for x, y in zip(a["images"], b["images"]):
        np.testing.assert_allclose(x, y, rtol=_order_bound(st["peeloffs"]), atol=0)
    np.testing.assert_allclose(a["absorption"], b["absorption"], rtol=_order_bound(st["path_crossings"]), atol=0)
    np.testing.assert_allclose(a["stats"], b["stats"], rtol=_order_bound(st["path_crossings"] + st["events"]), atol=0)


def _grid_problem(grid):
    if grid == "cartesian":
        return W.disk_galaxy(n_cells=24, n_lambda=2, n_pix=24, channels=3)
    if grid == "rectilinear":
        base = W.disk_galaxy(n_cells=4, n_lambda=2, n_pix=24, channels=3)
        edges = [W.powcub_edges(-25.0, 25.0, 17, 20.0), W.powcub_edges(-25.0, 25.0, 12, 20.0),
                 W.powcub_edges(-3.0, 3.0, 9, 50.0)]
        dens = np.random.default_rng(2).uniform(0.0, 2.0, (9, 12, 17))
        return W.replace(base, grid=W.rectilinear_grid(edges, dens))
    if grid == "octree":
        return W.clumpy_octree(n_particles=2000, n_samples=60_000, target_leaves=3000, max_level=6, n_lambda=2, n_pix=24)
    if grid == "bintree":
        return W.clumpy_bintree(n_particles=2000, n_samples=60_000, target_leaves=3000, max_level=6, n_lambda=2, n_pix=24)
    return W.voronoi_disk(n_sites=700, n_lambda=2, n_pix=24)


@pytest.mark.parametrize("views", ["frames", "shared"])
@pytest.mark.parametrize("grid", ["cartesian", "rectilinear", "octree", "bintree", "voronoi"])
def test_sorted_pass_equals_inline_walks(grid, views):
    """'shared': a second frame (other pixels and channels) and an SED of each of
    the problem's views, which take their optical depth from the first frame's
    record; 'frames': the problem's own.  The first launch sizes the record
    buffer, the second runs with the size from its count."""
    prob = _grid_problem(grid)
    if views == "shared":
        more = [dataclasses.replace(f, nx=7, ny=5, channels=3, bilinear=not f.bilinear) for f in prob.instruments]
        more += [dataclasses.replace(f, nx=1, ny=1, channels=1, bilinear=False, sed=True) for f in prob.instruments]
        prob = W.replace(prob, instruments=prob.instruments + more)
    n = 2500
    ref = PAR.gpu_run(prob, n, inline_peels=1, walk_peels=1)
    assert ref["raw_stats"]["sorted_peels"] == 0
    sim = rt.Simulation(prob)
    try:
        for k in range(2):
            sim.reset()
            got = PAR.gpu_run(prob, n, sim=sim, walk_peels=1)
            _assert_same(got, ref)
            st = got["raw_stats"]
            assert st["sorted_peels"] > 0
        assert st["sorted_peels"] == st["peeloffs"] - st["column_peels"]
    finally:
        sim.close()


@pytest.mark.parametrize("grid", ["rectilinear", "octree", "bintree", "voronoi"])
def test_launches_captured_into_a_graph(grid):
    """A launch recorded into a CUDA graph walks its peel-offs in place: two
    replays add up to two launches, and a plain launch afterwards takes the
    sorted pass again."""
    prob = _grid_problem(grid)
    n = 700
    ref = PAR.gpu_run(prob, n, walk_peels=1)
    sim = rt.Simulation(prob)
    try:
        sim.launch(n, walk_peels=1)  # the first launch of a problem makes its tables
        sim.reset()
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            sim.launch(n, 0, None, stream=torch.cuda.current_stream().cuda_stream, walk_peels=1)
        for k in range(2):
            graph.replay()
        torch.cuda.synchronize()
        st = sim.stats()
        assert st["device_flags"] == 0 and st["sorted_peels"] == 0
        assert st["peeloffs"] == 2 * ref["raw_stats"]["peeloffs"] and st["crossings"] == 2 * ref["raw_stats"]["crossings"]
        for x, y in zip(sim.images(), ref["images"]):
            np.testing.assert_allclose(x.cpu().numpy(), 2.0 * y, rtol=_order_bound(st["peeloffs"]), atol=0)
        sim.reset()
        again = PAR.gpu_run(prob, n, sim=sim, walk_peels=1)
        assert again["raw_stats"]["sorted_peels"] > 0
        for x, y in zip(again["images"], ref["images"]):
            np.testing.assert_allclose(x, y, rtol=_order_bound(st["peeloffs"]), atol=0)
    finally:
        sim.close()


@pytest.mark.parametrize("grid", ["cartesian", "octree"])
def test_launch_sizes_around_the_slots(grid):
    """Packets per wavelength from one to beyond every slot of the device: one
    warp, spread over the warps, each warp's slots full, and refilled.  Each
    launch equals the sum of two launches over its halves of the packet ids."""
    if grid == "cartesian":
        prob = W.uniform_cube(n_cells=6, axis_tau=2.0, n_pix=8)
    else:
        prob = W.clumpy_octree(n_particles=500, n_samples=5000, target_leaves=300, max_level=4, n_lambda=1, n_pix=8)
    warps = torch.cuda.get_device_properties(0).multi_processor_count * 8 * 4
    sim = rt.Simulation(prob)
    try:
        for n in (1, 2, 31, 33, warps - 1, warps + 1, 31 * warps + 1, 48 * warps - 1, 48 * warps + 1, 60 * warps - 1,
                  60 * warps + 1, 64 * warps + 33):
            sim.reset()
            one = PAR.gpu_run(prob, n, sim=sim)
            sim.reset()
            half = n // 2
            if half:
                sim.launch(half, 0, None, n_norm=n)
            two = PAR.gpu_run(prob, n - half, first_id=half, sim=sim, n_norm=n)
            assert one["counters"][3] == n
            _assert_same(one, two)
    finally:
        sim.close()


def test_batch_models_around_the_run_lengths():
    """A batch's warps take runs of 64 to 1024 packets of one model: models of
    fewer packets than a run, of a run and its neighbours, and of many runs."""
    counts = [1, 63, 64, 65, 1023, 1025, 40_000]
    allm = W.batch_models()
    probs = [W.with_packets(allm[i], c) for i, c in enumerate(counts)]
    b = rt.Batch(probs)
    try:
        b.launch(seed=3)
        imgs, st = b.images(), b.stats()
    finally:
        b.close()
    assert st["device_flags"] == 0 and st["packets"] == sum(counts)
    for m, (p, c) in enumerate(zip(probs, counts)):
        sim = rt.Simulation(p)
        try:
            sim.launch(c, 0, 3, model_id=m)
            one = sim.stats()
            np.testing.assert_allclose(imgs[m], sim.images(device=False)[0][0, 0], rtol=_order_bound(one["peeloffs"]), atol=0)
        finally:
            sim.close()
