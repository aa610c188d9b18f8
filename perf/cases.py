"""The work that users of the transport library have it do, as timed cases.

Every case goes through the public Python entry points (``rt.Simulation``,
``rt.Batch``, ``autograd.transport``, the ``rt_*`` calls): what a program keeps
between calls (contexts with their grid, optics, sources and instruments) is
made by :func:`prepare`, one pass of its inner loop is :func:`run`.  Sizes and
settings are those of the workloads, tests and benchmark of this repository,
scaled to a fraction of a second.
"""
import functools
import math

import numpy as np
import torch

from paper_1410_1629_gb300 import rt
from paper_1410_1629_gb300 import workloads as W
from paper_1410_1629_gb300.autograd import transport


def listed():
    return [
        # A look at a small model while its parameters are tried out: the
        # latency of one call is all that counts.
        dict(name="cube_preview", kind="cube", cells=32, packets=10_000, pix=64, tau=1.0, albedo=0.6),
        # A galaxy model of ordinary size with no round dimension: frames
        # along and across the grid, total / direct / scattered channels and
        # an SED, results taken to the host.
        dict(name="disk_ragged", kind="disk", nx=101, ny=77, nz=45, n_lambda=3, packets=300_000, pix=83, channels=3,
             sed=True, host=True),
        # The production run: the edge-on disk galaxy of the benchmark (256^3
        # cells, 10 wavelengths, three frames).
        dict(name="disk_galaxy", kind="disk", nx=256, ny=256, nz=256, n_lambda=10, packets=20_000_000, pix=512,
             channels=1, sed=False, host=False),
        # The paper's worked example on its power-law grid.
        dict(name="spiral_powcub", kind="spiral", n_xy=256, n_z=128, packets=4_000_000, pix=1200, pix_y=300),
        # Clumpy dust on the adaptive grids: octree, k-d tree, Voronoi.
        dict(name="octree_clumpy", kind="octree", leaves=400_000, level=9, n_lambda=5, packets=2_000_000, pix=256),
        dict(name="bintree_clumpy", kind="bintree", leaves=200_000, level=8, n_lambda=4, packets=2_000_000, pix=512),
        dict(name="voronoi_disk", kind="voronoi", sites=30_000, n_lambda=3, packets=1_500_000, pix=256),
        # A parameter search: many small models in one launch.
        dict(name="batch_search", kind="batch", models=256, pix=64),
        # One step of fitting a density to an image: forward with the adjoint
        # tape and the gradient; and the same with an absorption target,
        # whose gradient replays the packets.
        dict(name="fit_image", kind="fit", cells=64, packets=1_000_000, pix=128, events=20, absorption=False),
        dict(name="fit_absorption", kind="fit", cells=48, packets=200_000, pix=64, events=20, absorption=True),
        # Panchromatic mode: the dust's equilibrium temperatures and thermal
        # emission from a given absorption field, and a whole iteration
        # (stars, temperatures, emission table, dust).
        dict(name="dust_temperature", kind="dust", nx=192, ny=192, nz=128, n_lambda=24),
        dict(name="panchromatic", kind="panchromatic", cells=96, n_lambda=24, packets=1_200_000, pix=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cube", "disk", "disk", "spiral", "octree", "bintree", "voronoi", "batch", "fit", "fit", "dust",
                       "panchromatic"])
    if kind == "cube":
        return dict(kind=kind, cells=rng.randint(8, 64), packets=_log_int(rng, 2_000, 2_000_000),
                    pix=rng.randint(16, 128), tau=round(rng.uniform(0.1, 10.0), 3), albedo=round(rng.uniform(0.1, 0.9), 3))
    if kind == "disk":
        return dict(kind=kind, nx=_log_int(rng, 32, 256), ny=_log_int(rng, 32, 256), nz=_log_int(rng, 16, 200),
                    n_lambda=rng.randint(1, 8), packets=_log_int(rng, 50_000, 6_000_000), pix=_log_int(rng, 32, 512),
                    channels=rng.choice([1, 3]), sed=rng.random() < 0.5, host=rng.random() < 0.3)
    if kind == "spiral":
        return dict(kind=kind, n_xy=rng.randint(48, 256), n_z=rng.randint(32, 128),
                    packets=_log_int(rng, 100_000, 4_000_000), pix=rng.randint(200, 1200), pix_y=rng.randint(60, 300))
    if kind in ("octree", "bintree"):
        return dict(kind=kind, leaves=_log_int(rng, 10_000, 400_000), level=rng.randint(7, 9), n_lambda=rng.randint(1, 6),
                    packets=_log_int(rng, 50_000, 1_500_000), pix=rng.randint(48, 512))
    if kind == "voronoi":
        return dict(kind=kind, sites=_log_int(rng, 2_000, 30_000), n_lambda=rng.randint(1, 3),
                    packets=_log_int(rng, 30_000, 1_500_000), pix=rng.randint(48, 256))
    if kind == "batch":
        return dict(kind=kind, models=_log_int(rng, 16, 256), pix=rng.randint(24, 64))
    if kind == "fit":
        absorption = rng.random() < 0.4
        return dict(kind=kind, cells=rng.randint(12, 64), packets=_log_int(rng, 20_000, 250_000 if absorption else 1_000_000),
                    pix=rng.randint(16, 128), events=rng.randint(5, 20), absorption=absorption)
    if kind == "dust":
        return dict(kind=kind, nx=_log_int(rng, 24, 192), ny=_log_int(rng, 24, 192), nz=_log_int(rng, 16, 128),
                    n_lambda=rng.randint(8, 24))
    return dict(kind=kind, cells=rng.randint(32, 96), n_lambda=rng.randint(8, 24), packets=_log_int(rng, 100_000, 1_200_000),
                pix=rng.randint(24, 128))


# ---------------------------------------------------------------- problems
@functools.lru_cache(maxsize=4)
def _tree(kind, leaves, level, n_lambda, pix):
    """The refined grid of the clumpy medium; its density varies with the seed."""
    make = W.clumpy_octree if kind == "octree" else W.clumpy_bintree
    return make(n_particles=max(2_000, leaves // 4), n_samples=25 * leaves, target_leaves=leaves, max_level=level,
                n_lambda=n_lambda, n_pix=pix)


@functools.lru_cache(maxsize=4)
def _voronoi(sites, n_lambda, pix):
    return W.voronoi_disk(n_sites=sites, n_lambda=n_lambda, n_pix=pix)


@functools.lru_cache(maxsize=4)
def _spiral(n_xy, n_z, pix, pix_y):
    return W.spiral_example("powcub", n_xy=n_xy, n_z=n_z, n_pix=(pix, pix_y))


def _disk_grid(shape):
    bounds = [-25.0, 25.0, -25.0, 25.0, -3.0, 3.0]
    xs, ys, zs = W.cell_centres(bounds, shape)
    R = np.sqrt(xs[None, :] ** 2 + ys[:, None] ** 2)
    dens = np.exp(-np.abs(zs) / 0.2)[:, None, None].astype(np.float32) * np.exp(-R / 6.0)[None].astype(np.float32)
    return W.cartesian_grid(bounds, dens)


def _problem(case, seed):
    """The model of a case: the workload's grid with every cell's density
    scaled by a log-normal factor of 10 % drawn from the seed."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "cube":
        p = W.uniform_cube(n_cells=case["cells"], n_pix=case["pix"], axis_tau=case["tau"], albedo=case["albedo"],
                           source_pos=tuple(rng.uniform(-0.2, 0.2, 3)))
    elif kind in ("disk", "panchromatic", "dust"):
        if kind == "disk":
            shape = (case["nx"], case["ny"], case["nz"])
            p = W.disk_galaxy(n_cells=2, n_lambda=case["n_lambda"], n_pix=case["pix"], channels=case["channels"])
            if case["sed"]:
                p = W.replace(p, instruments=p.instruments + [W.sed_instrument(60.0, channels=case["channels"])])
        else:
            shape = (case["cells"],) * 3 if kind == "panchromatic" else (case["nx"], case["ny"], case["nz"])
            p = W.panchromatic_disk(n_cells=2, n_lambda=case["n_lambda"], n_pix=case.get("pix", 8))
        p = W.replace(p, grid=_disk_grid(shape))
    elif kind == "spiral":
        p = _spiral(case["n_xy"], case["n_z"], case["pix"], case["pix_y"])
    elif kind in ("octree", "bintree"):
        p = _tree(kind, case["leaves"], case["level"], case["n_lambda"], case["pix"])
    elif kind == "voronoi":
        p = _voronoi(case["sites"], case["n_lambda"], case["pix"])
    elif kind == "fit":
        p = W.lognormal_cube(n_cells=case["cells"], n_pix=case["pix"], max_events=case["events"], seed=seed % 100_000)
    dens = p.grid.density
    noise = rng.standard_normal(dens.shape, dtype=np.float32)
    noise *= np.float32(0.1)
    p = W.with_density(p, dens * np.exp(noise, out=noise))
    return W.with_packets(p, max(1, case["packets"] // p.n_lambda)) if "packets" in case else p


# constants of the thermal emission (the library's reading: lambda^-5 / (exp(C2 / lambda T) - 1))
_C2 = 14387.768775039337


def _dust_weights(p):
    """a_l, b_l of the emission per unit mass sum_l a_l / (exp(b_l / T) - 1)."""
    lam = np.asarray(p.wavelengths, dtype=np.float64)
    mid = np.sqrt(lam[1:] * lam[:-1])
    edges = np.concatenate([[lam[0] * math.sqrt(lam[0] / lam[1])], mid, [lam[-1] * math.sqrt(lam[-1] / lam[-2])]])
    return p.meta["emission_scale"] * p.kappa * (1.0 - p.albedo) * np.diff(edges) / lam ** 5, _C2 / lam


def _cell_mass(p, device):
    """rho V per row-major cell, float64."""
    b = np.asarray(p.grid.bounds, dtype=np.float64)
    n = p.grid.shape
    d = [np.diff(b[2 * a] + np.arange(n[a] + 1) * ((b[2 * a + 1] - b[2 * a]) / n[a])) for a in range(3)]
    vol = d[2][:, None, None] * d[1][None, :, None] * d[0][None, None, :]
    return torch.from_numpy(p.grid.density.reshape(-1)).to(device).double() * torch.from_numpy(vol.reshape(-1)).to(device)


def _per_mass(a, b, T):
    out = torch.zeros_like(T)
    for al, bl in zip(a, b):
        out += al / torch.expm1(bl / T)
    return out


def _absorbed_field(p, seed, device):
    """An absorption field [n_lambda, n_cells] whose dust settles at 4 to 60
    K, warm in the middle, with 5 % of the cells untouched by any packet."""
    g = torch.Generator(device=device).manual_seed(seed)
    m = _cell_mass(p, device)
    n = m.numel()
    rho = torch.from_numpy(p.grid.density.reshape(-1)).to(device).double()
    u = torch.rand(n, generator=g, device=device, dtype=torch.float64)
    T0 = 4.0 + 40.0 * rho.clamp(max=1.2) + 8.0 * u
    a, b = _dust_weights(p)
    total = m * _per_mass(a, b, T0)
    total[torch.rand(n, generator=g, device=device) < 0.05] = 0.0
    share = torch.from_numpy(np.asarray(p.sources[0].lum * p.kappa * (1.0 - p.albedo))).to(device)
    return (share / share.sum())[:, None] * total[None, :]


# ---------------------------------------------------------------- the cases
def prepare(case, seed):
    kind = case["kind"]
    state = dict(case=case, seed=seed % (1 << 31))
    if kind == "batch":
        models = W.batch_models(n_models=case["models"], n_pix=case["pix"], seed=seed)
        return dict(state, batch=rt.Batch(models))
    p = _problem(case, seed)
    state["sim"] = sim = rt.Simulation(p)
    device = torch.device("cuda", sim.device)
    if kind == "fit":
        state["density"] = torch.from_numpy(p.grid.density).to(device).requires_grad_(True)
        g = torch.Generator(device=device).manual_seed(seed)
        state["target"] = [0.02 * torch.rand(sim.image_shape(q), generator=g, device=device, dtype=torch.float64) / case["pix"]
                           for q in range(len(p.instruments))]
        state["target_absorption"] = torch.rand((1, p.grid.n_cells), generator=g, device=device, dtype=torch.float64) / p.grid.n_cells
    if kind == "dust":
        state["absorbed"] = _absorbed_field(p, seed, device)
        state["T"] = torch.zeros(p.grid.n_cells, dtype=torch.float64, device=device)
        state["emission"] = torch.zeros((p.n_lambda, p.grid.n_cells), dtype=torch.float64, device=device)
        torch.cuda.synchronize()
    return state


def run(state):
    case, seed = state["case"], state["seed"]
    kind = case["kind"]
    if kind == "batch":
        b = state["batch"]
        b.reset()
        b.launch(seed)
        return {"images": b.images_flat(), "tallies": b.tallies()}
    sim = state["sim"]
    if kind == "fit":
        density = state["density"]
        images, absorption = transport(density, sim, seed=seed)
        outputs, residuals = list(images), [i - t for i, t in zip((i.detach() for i in images), state["target"])]
        if case["absorption"]:
            outputs.append(absorption)
            residuals.append(absorption.detach() - state["target_absorption"])
        (grad,) = torch.autograd.grad(outputs, density, residuals)
        return {"images": [i.detach() for i in images], "absorption": absorption.detach(), "grad": grad}
    if kind == "dust":
        S = sim.problem.meta["emission_scale"]
        T, out = state["T"], state["emission"]
        held = rt.rt_dust_temperature(sim.ctx, S, 1.0, 1e4, state["absorbed"].data_ptr(), 1, T.data_ptr(), 1)
        rt.rt_set_dust_emission(sim.ctx, T.data_ptr(), 1, S)
        rt.rt_read_dust_emission(sim.ctx, out.data_ptr(), out.numel(), 1)
        return {"temperature": T, "emission": out, "held": held}
    sim.reset()
    sim.launch(seed=seed)
    if kind == "panchromatic":
        S = sim.problem.meta["emission_scale"]
        stars = sim.images()
        T, held = sim.dust_temperature(S)
        sim.set_dust_emission(T, S)
        sim.reset()
        sim.launch(seed=seed + 1, emitter=rt.RT_EMITTER_DUST)
        return {"stars": stars, "temperature": T, "held": held, "dust": sim.images(), "absorption": sim.absorption()}
    device = not case.get("host", False)
    return {"images": sim.images(device=device), "absorption": sim.absorption(device=device)}


# ---------------------------------------------------------------- the work
# Floating-point operations of one cell crossing: three plane parameters and
# their minimum, the segment, the optical depth and an exponential.
_CROSSING = 24


def _path_work(cells_on_path, packets, events, walked_frames):
    """Operations of the packets' walks: per event one forced path and the
    half of it up to the interaction, and a half path per walked frame."""
    return _CROSSING * packets * events * cells_on_path * (1.5 + 0.5 * walked_frames)


def work(case):
    kind = case["kind"]
    packets = case.get("packets", 0)
    pix = case.get("pix", 0)
    if kind == "batch":
        models = W.batch_models(n_models=case["models"], n_pix=case["pix"])
        cells = sum(m.grid.n_cells for m in models)
        flops = sum(_path_work(m.grid.shape[0], m.run.n_per_lambda, 4, 0) for m in models)
        return {"bytes": 4 * cells + 8 * case["models"] * (pix * pix + 4), "flops": flops}
    if kind == "cube":
        n = case["cells"] ** 3
        return {"bytes": 12 * n + 8 * pix * pix, "flops": _path_work(case["cells"], packets, 6, 0)}
    if kind == "disk":
        n = case["nx"] * case["ny"] * case["nz"]
        image = 8 * case["n_lambda"] * case["channels"] * (3 * pix * pix + (1 if case["sed"] else 0))
        path = 0.3 * (case["nx"] + case["ny"]) + 0.5 * case["nz"]
        return {"bytes": 4 * n + 8 * case["n_lambda"] * n + image,
                "flops": _path_work(path, packets, 4, 2 if case["sed"] else 1)}
    if kind == "spiral":
        n = case["n_xy"] ** 2 * case["n_z"]
        return {"bytes": 12 * n + 8 * pix * case["pix_y"], "flops": _path_work(case["n_xy"], packets, 4, 0)}
    if kind in ("octree", "bintree"):
        n = case["leaves"]
        return {"bytes": 8 * n + 8 * case["n_lambda"] * n + 16 * case["n_lambda"] * pix * pix,
                "flops": _path_work(1.2 * n ** (1 / 3), packets, 4, 2)}
    if kind == "voronoi":
        n = case["sites"]
        return {"bytes": (28 + 20 * 15) * n + 8 * case["n_lambda"] * n + 24 * case["n_lambda"] * pix * pix,
                "flops": 5 * _path_work(1.5 * n ** (1 / 3), packets, 4, 3)}
    if kind == "fit":
        n = case["cells"] ** 3
        forward = _path_work(1.2 * case["cells"], packets, case["events"], 0)
        return {"bytes": 4 * n + 8 * n + 4 * n + 16 * pix * pix + (8 * n if case["absorption"] else 0),
                "flops": (2.5 if case["absorption"] else 1.7) * forward}
    nl = case["n_lambda"]
    if kind == "dust":
        n = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": n * (8 * nl + 4 + 8 + 8 * nl), "flops": 40.0 * n * nl}
    n = case["cells"] ** 3
    return {"bytes": n * (2 * (4 + 8 * nl) + 16 + 8 * nl) + 2 * 8 * nl * 3 * pix * pix,
            "flops": 2 * _path_work(1.1 * case["cells"], packets, 3, 2) + 40.0 * n * nl}


# ---------------------------------------------------------------- 64-bit values
def exact(case, seed):
    """The same packets followed in 64 bits by plain torch (grids of equal
    cells, launches small enough for it), or the dust's temperatures and
    emission by bisection; None for the trees, the Voronoi grid, batches and
    the large launches."""
    kind = case["kind"]
    device = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if kind == "dust":
        p = _problem(case, seed)
        T = _temperature64(p, _absorbed_field(p, seed, device))
        a, b = _dust_weights(p)
        m = _cell_mass(p, device)
        emission = torch.stack([torch.where(T > 0, m * (al / torch.expm1(bl / T)), 0.0) for al, bl in zip(a, b)])
        return {"temperature": T, "emission": emission, "held": None}
    if kind not in ("cube", "disk", "fit") or case["packets"] * case.get("n_lambda", 1) > 1_200_000:
        return None
    images, absorption = _transport64(_problem(case, seed), seed % (1 << 31), device)
    out = {"images": images, "absorption": absorption}
    if kind == "fit":
        out["grad"] = None
    elif case.get("host"):
        out = {"images": [i.cpu().numpy() for i in images], "absorption": absorption.cpu().numpy()}
    return out


def _temperature64(p, absorbed):
    a, b = _dust_weights(p)
    m = _cell_mass(p, absorbed.device)
    total = torch.zeros_like(m)
    for row in absorbed:
        total += row
    lo, hi = torch.zeros_like(m), torch.full_like(m, math.log(1e4))  # ln of 1 K and 1e4 K
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        low = m * _per_mass(a, b, mid.exp()) < total
        lo, hi = torch.where(low, mid, lo), torch.where(low, hi, mid)
    return torch.where((total > 0) & (m > 0), (0.5 * (lo + hi)).exp(), 0.0)


_M32 = 0xFFFFFFFF


def _philox(ids, lam, event, block, seed):
    """Philox4x32-10 (Salmon et al. 2011): counter (id low, id high, event,
    lambda << 8 | block), key (seed, 0); four 32-bit words as int64."""
    def mul(const, v):  # high and low word of a 32 x 32 bit product
        p, q = const * (v & 0xFFFF), const * (v >> 16)
        low = p + ((q & 0xFFFF) << 16)
        return (q >> 16) + (low >> 32), low & _M32
    c = [ids & _M32, ids >> 32, torch.full_like(ids, event), (lam << 8) | block]
    k0, k1 = seed & _M32, 0
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return [(v.double() + 0.5) * 2.0 ** -32 for v in c]


class _Grid64:
    def __init__(self, p, device):
        b = np.asarray(p.grid.bounds, dtype=np.float64)
        self.n = torch.tensor(p.grid.shape, device=device)
        self.lo = torch.tensor(b[0::2], device=device)
        self.hi = torch.tensor(b[1::2], device=device)
        self.d = (self.hi - self.lo) / self.n
        self.rho = torch.from_numpy(p.grid.density.reshape(-1)).to(device).double()

    def cell_id(self, i):
        return i[:, 0] + self.n[0] * (i[:, 1] + self.n[1] * i[:, 2])

    def walk(self, x, k, kappa, cell=None, stop=None, deposit=None):
        """Optical depth from x along k to the boundary; with `stop` the cell
        and distance at which it is reached; `deposit(rows, cell, tau, dtau)`
        sees every segment."""
        N = len(x)
        tau_all = torch.zeros(N, dtype=torch.float64, device=x.device)
        hit_cell, hit_t = torch.zeros((N, 3), dtype=torch.int64, device=x.device), torch.zeros_like(tau_all)
        inv = torch.where(k != 0, 1.0 / k, math.inf)
        t = torch.zeros_like(tau_all)
        rows = torch.arange(N, device=x.device)
        if cell is None:
            t1, t2 = (self.lo - x) * inv, (self.hi - x) * inv
            near = torch.where(k != 0, torch.minimum(t1, t2), -math.inf)
            far = torch.where(k != 0, torch.maximum(t1, t2), math.inf)
            inside = ((x >= self.lo) & (x <= self.hi)).all(1)
            parallel_out = ((k == 0) & ((x < self.lo) | (x > self.hi))).any(1)
            t_in, t_out = near.amax(1), far.amin(1)
            ok = inside | ((t_in < t_out) & (t_out > 0) & ~parallel_out)
            t = torch.where(inside, 0.0, t_in)
            at = x + torch.where(ok, t, 0.0)[:, None] * k
            cell = torch.minimum(torch.floor((at - self.lo) / self.d).long().clamp(min=0), self.n - 1)
            rows = rows[ok]
        x, k, inv, t, i, kap = x[rows], k[rows], inv[rows], t[rows], cell[rows], kappa[rows]
        goal = stop[rows] if stop is not None else None
        tau = torch.zeros_like(t)
        up, step = (k > 0).long(), torch.sign(k).long()
        while len(rows):
            plane = self.lo + (i + up) * self.d
            t_exit, axis = torch.where(k != 0, (plane - x) * inv, math.inf).min(1)
            t_exit = torch.maximum(t_exit, t)
            c = self.cell_id(i)
            kr = kap * self.rho[c]
            dt = kr * (t_exit - t)
            if deposit is not None:
                deposit(rows, c, tau, dt)
            nxt = tau + dt
            alive = torch.ones_like(rows, dtype=torch.bool)
            if goal is not None:
                hit = nxt > goal
                hit_cell[rows[hit]] = i[hit]
                hit_t[rows[hit]] = (t + (goal - tau) / kr)[hit]
                alive = ~hit
            j = i.scatter_add(1, axis[:, None], step.gather(1, axis[:, None]))
            out = ((j < 0) | (j >= self.n)).any(1)
            if goal is not None:  # rounding: kept at the end of the path
                last = out & alive
                hit_cell[rows[last]], hit_t[rows[last]] = i[last], t_exit[last]
            gone = out | ~alive
            tau_all[rows[gone]] = nxt[gone]
            keep = ~gone
            x, k, inv, i, kap, rows, t, tau = x[keep], k[keep], inv[keep], j[keep], kap[keep], rows[keep], t_exit[keep], nxt[keep]
            up, step = up[keep], step[keep]
            goal = goal[keep] if goal is not None else None
        return tau_all, hit_cell, hit_t


def _rotated(k, mu, phi):
    st = torch.sqrt((1 - mu * mu).clamp(min=0))
    s = torch.sqrt(k[:, 0] ** 2 + k[:, 1] ** 2)
    safe = torch.where(s > 0, s, 1.0)
    cx, cy = k[:, 0] / safe, k[:, 1] / safe
    cp, sp = torch.cos(phi), torch.sin(phi)
    n = torch.stack([mu * k[:, 0] + st * (cp * cx * k[:, 2] - sp * cy), mu * k[:, 1] + st * (cp * cy * k[:, 2] + sp * cx),
                     mu * k[:, 2] - st * cp * s], 1)
    z = torch.sign(k[:, 2])
    pole = torch.stack([st * cp, z * st * sp, z * mu], 1)
    n = torch.where((s > 0)[:, None], n, pole)
    return n / n.norm(dim=1, keepdim=True)


def _snap(v):
    return float(round(v)) if abs(v - round(v)) < 1e-15 else v


def _transport64(p, seed, device):
    grid = _Grid64(p, device)
    n, nl = p.run.n_per_lambda, p.n_lambda
    ids = torch.arange(n, device=device).repeat(nl)
    lam = torch.arange(nl, device=device).repeat_interleave(n)
    table = [torch.tensor(np.asarray(v, dtype=np.float64), device=device) for v in (p.kappa, p.albedo, p.g, p.sources[0].lum)]
    kappa, albedo, g = (v[lam] for v in table[:3])
    L0 = table[3][lam] / n
    absorption = torch.zeros(nl * p.grid.n_cells, dtype=torch.float64, device=device)
    frames, images = [], []
    for q in p.instruments:
        si, ci, sa, ca = (_snap(f(v)) for v in (q.inclination, q.azimuth) for f in (math.sin, math.cos))
        so, co = _snap(math.sin(q.position_angle)), _snap(math.cos(q.position_angle))
        a, b = np.array([-sa, ca, 0.0]), np.array([-ci * ca, -ci * sa, si])
        frames.append([torch.tensor(v, device=device, dtype=torch.float64)
                       for v in ([si * ca, si * sa, ci], co * a - so * b, so * a + co * b)])
        images.append(torch.zeros((q.channels, nl, q.ny, q.nx), dtype=torch.float64, device=device))

    def peel(x, cell, lam, kappa, L, k, g, channel):
        for q, (kobs, ex, ey), image in zip(p.instruments, frames, images):
            tau, _, _ = grid.walk(x, kobs.expand(len(x), 3), kappa, cell)
            phase = 1.0
            if channel == 2:
                mu = k @ kobs
                phase = (1 - g * g) / (1 + g * g - 2 * g * mu) ** 1.5
            value = L * phase * torch.exp(-tau) / (4 * math.pi)
            flat = image.view(q.channels, -1)
            spots = [(torch.zeros_like(lam), torch.zeros_like(lam), 1.0)]
            if not q.sed:
                fx = (x @ ex + q.half_x - q.center_x) * (q.nx / (2 * q.half_x))
                fy = (x @ ey + q.half_y - q.center_y) * (q.ny / (2 * q.half_y))
                spots = [(torch.floor(fx).long(), torch.floor(fy).long(), 1.0)]
                if q.bilinear:
                    x0, y0 = torch.floor(fx - 0.5), torch.floor(fy - 0.5)
                    tx, ty = fx - 0.5 - x0, fy - 0.5 - y0
                    spots = [(x0.long() + dx, y0.long() + dy, (tx if dx else 1 - tx) * (ty if dy else 1 - ty))
                             for dx in (0, 1) for dy in (0, 1)]
            for px, py, w in spots:
                ok = (px >= 0) & (py >= 0) & (px < q.nx) & (py < q.ny)
                at = ((lam * q.ny + py) * q.nx + px)[ok]
                for ch in ([0, channel] if q.channels == 3 else [0]):
                    flat[ch].index_add_(0, at, (value * w)[ok])

    # emission
    r0, r1 = _philox(ids, lam, 0, 0, seed), _philox(ids, lam, 0, 1, seed)
    s = p.sources[0]
    x = torch.tensor(s.center, dtype=torch.float64, device=device).repeat(len(ids), 1)
    if s.kind == "expdisk":
        R = -s.scale_r * (torch.log(r0[1]) + torch.log(r0[2]))
        z = -s.scale_z * torch.log(r1[0])
        phi = 2 * math.pi * r0[3]
        x = x + torch.stack([R * torch.cos(phi), R * torch.sin(phi), torch.where(r1[1] < 0.5, -z, z)], 1)
    mu, phi = 2 * r1[2] - 1, 2 * math.pi * r1[3]
    st = torch.sqrt(1 - mu * mu)
    k = torch.stack([st * torch.cos(phi), st * torch.sin(phi), mu], 1)
    L, cell = L0.clone(), None
    peel(x, None, lam, kappa, L, k, g, 1)
    for event in range(1, p.run.max_events + 1):
        def deposit(rows, c, tau, dt):
            absorption.index_add_(0, lam[rows] * p.grid.n_cells + c,
                                  ((1 - albedo) * L)[rows] * torch.exp(-tau) * -torch.expm1(-dt))
        tau, _, _ = grid.walk(x, k, kappa, cell, deposit=deposit)
        on = tau > 0
        ids, lam, kappa, albedo, g, L0, x, k, L, tau = (v[on] for v in (ids, lam, kappa, albedo, g, L0, x, k, L, tau))
        cell = cell[on] if cell is not None else None
        if not len(ids):
            break
        r = _philox(ids, lam, event, 0, seed)
        part = -torch.expm1(-tau)
        _, cell, s_star = grid.walk(x, k, kappa, cell, stop=-torch.log1p(-r[0] * part))
        L = albedo * L * part
        x = x + s_star[:, None] * k
        x = torch.minimum(torch.maximum(x, grid.lo + cell * grid.d), grid.lo + (cell + 1) * grid.d)
        peel(x, cell, lam, kappa, L, k, g, 2)
        small = g.abs() < 1e-6
        gs = torch.where(small, 0.5, g)
        f = (1 - gs * gs) / (1 - gs + 2 * gs * r[1])
        mu = torch.where(small, 2 * r[1] - 1, ((1 + gs * gs - f * f) / (2 * gs)).clamp(-1, 1))
        k = _rotated(k, mu, 2 * math.pi * r[2])
        on = L >= p.run.w_min * L0 if p.run.weight_cut else torch.ones_like(lam, dtype=torch.bool)
        ids, lam, kappa, albedo, g, L0, x, k, L, cell = (v[on] for v in (ids, lam, kappa, albedo, g, L0, x, k, L, cell))
    return images, absorption.view(nl, -1)
