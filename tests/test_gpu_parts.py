"""The sorted peel-off pass with a record buffer that is small by choice
(part_records): launches in several parts, whose borders fall inside a
wavelength, and buffers that overflow, so that part of the peel-offs walk in
place, give what walking every peel-off in place gives.  Two routes add the same
positive FP64 contributions in different orders: a sum of n of them differs by at
most 2 n 2^-53 relative."""
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

GRIDS = ["cartesian", "rectilinear", "octree", "bintree", "voronoi"]


def _problem(grid, shared):
    if grid == "cartesian":
        prob = W.disk_galaxy(n_cells=24, n_lambda=3, n_pix=24, channels=3)
    elif grid == "rectilinear":
        edges = [W.powcub_edges(-25.0, 25.0, 17, 20.0), W.powcub_edges(-25.0, 25.0, 12, 20.0),
                 W.powcub_edges(-3.0, 3.0, 9, 50.0)]
        dens = np.random.default_rng(2).uniform(0.0, 2.0, (9, 12, 17))
        prob = W.replace(W.disk_galaxy(n_cells=4, n_lambda=3, n_pix=24, channels=3), grid=W.rectilinear_grid(edges, dens))
    elif grid == "octree":
        prob = W.clumpy_octree(n_particles=2000, n_samples=60_000, target_leaves=3000, max_level=6, n_lambda=3, n_pix=24)
    elif grid == "bintree":
        prob = W.clumpy_bintree(n_particles=2000, n_samples=60_000, target_leaves=3000, max_level=6, n_lambda=3, n_pix=24)
    else:
        prob = W.voronoi_disk(n_sites=700, n_lambda=3, n_pix=24)
    if shared:  # a second frame and an SED of every view: they share the first frame's records
        more = [dataclasses.replace(f, nx=7, ny=5, channels=3, bilinear=not f.bilinear) for f in prob.instruments]
        more += [dataclasses.replace(f, nx=1, ny=1, channels=1, bilinear=False, sed=True) for f in prob.instruments]
        prob = W.replace(prob, instruments=prob.instruments + more)
    return prob


def _assert_same(a, b):
    assert np.array_equal(a["counters"], b["counters"])
    st = a["raw_stats"]
    assert st["device_flags"] == b["raw_stats"]["device_flags"] == 0
    bound = lambda n: 2.0 * float(n) * 2.0 ** -53  # noqa: E731
    for x, y in zip(a["images"], b["images"]):
        np.testing.assert_allclose(x, y, rtol=bound(st["peeloffs"]), atol=0)
    np.testing.assert_allclose(a["absorption"], b["absorption"], rtol=bound(st["path_crossings"]), atol=0)
    np.testing.assert_allclose(a["stats"], b["stats"], rtol=bound(st["path_crossings"] + st["events"]), atol=0)


@pytest.mark.parametrize("shared", [False, True])
@pytest.mark.parametrize("grid", GRIDS)
def test_parts_and_overflow_equal_walks_in_place(grid, shared):
    prob = _problem(grid, shared)
    n = 2501  # packets per wavelength
    ref = PAR.gpu_run(prob, n, inline_peels=1, walk_peels=1)
    sim = rt.Simulation(prob)
    try:
        for records in (5000, 700, 1):  # parts of many packets, of few, of one (cartesian: walks in place from there)
            m = n if records > 1 else 40
            one = ref if m == n else PAR.gpu_run(prob, m, inline_peels=1, walk_peels=1)
            for _ in range(2):  # the first launch with an estimate of records per packet, the second with a count
                sim.reset()
                got = PAR.gpu_run(prob, m, sim=sim, walk_peels=1, part_records=records)
                _assert_same(got, one)
            sorted_peels = got["raw_stats"]["sorted_peels"]
            if grid == "cartesian":  # one part, its overflow in place
                assert records <= sorted_peels <= records * len(prob.instruments)
            else:  # more than one buffer's worth of records went through the pass (a record serves up to three)
                assert sorted_peels > 2 * records * (3 if shared else 1)
        for _ in range(2):  # the library's own limit again
            sim.reset()
            got = PAR.gpu_run(prob, n, sim=sim, walk_peels=1)
            _assert_same(got, ref)
        assert got["raw_stats"]["sorted_peels"] == ref["raw_stats"]["peeloffs"]
    finally:
        sim.close()


@pytest.mark.parametrize("shared", [False, True])
@pytest.mark.parametrize("grid", GRIDS)
def test_buffer_sized_by_a_launch_of_fewer_records(grid, shared):
    """A launch without scattering peel-offs leaves an estimate far too small for
    the next: its buffer overflows in every part, also between an instrument whose
    record still fits and those that would share it."""
    prob = _problem(grid, shared)
    n = 1203
    ref = PAR.gpu_run(prob, n, inline_peels=1, walk_peels=1)
    sim = rt.Simulation(prob)
    try:
        sim.launch(n, walk_peels=1, peel_scatter=0, part_records=3000)
        torch.cuda.synchronize()
        sim.reset()
        got = PAR.gpu_run(prob, n, sim=sim, walk_peels=1, part_records=1001)
        _assert_same(got, ref)
        assert 0 < got["raw_stats"]["sorted_peels"] < got["raw_stats"]["peeloffs"]
    finally:
        sim.close()


def test_no_small_parts_when_memory_is_short():
    """With memory for fewer than 2^23 of its records a launch walks its peel-offs in
    place; with memory given back it sorts them again."""
    prob = _problem("octree", False)
    n = 400_000  # of 3 wavelengths: 1.2e6 packets, 0.7 GB of records at the first estimate
    sim = rt.Simulation(prob)
    hold = None
    try:
        sim.launch(n, inline_peels=1)  # the kernels and tables are loaded
        ref = [t.cpu().numpy() for t in sim.images()]
        st_ref = sim.stats()
        sim.launch(10, inline_peels=0)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        hold = torch.empty(free - (500 << 20), dtype=torch.uint8, device="cuda")  # 0.2 GB of records fit
        sim.reset()
        sim.launch(n)
        st = sim.stats()
        assert st["device_flags"] == 0 and st["sorted_peels"] == 0
        assert st["crossings"] == st_ref["crossings"] and st["peeloffs"] == st_ref["peeloffs"]
        for x, y in zip(sim.images(), ref):
            np.testing.assert_allclose(x.cpu().numpy(), y, rtol=2.0 * st["peeloffs"] * 2.0 ** -53, atol=0)
        del hold
        hold = None
        torch.cuda.empty_cache()
        sim.reset()
        sim.launch(n)
        assert sim.stats()["sorted_peels"] == st_ref["peeloffs"]
    finally:
        del hold
        torch.cuda.empty_cache()
        sim.close()
