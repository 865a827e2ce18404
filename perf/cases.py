"""The work that a user of this framework has it do, as cases that can be timed.

A case is a dict of plain values: the call (``op``), the point cloud (``mesh``,
``points``) and the sizes of the line-transfer problem.  The clouds, line lists
and field laws are those of ``paper_2411_03040_gb300.synth`` (the laws of this
repository's benchmarks and tests).  The neighbour graph belongs to a cloud of
a given kind and size; the seed draws its orientation (every direction then
sees other rays), the scatter of the fields, the line data's collision rates
and the viewing directions.

``exact`` restates each path in plain torch in 64 bits.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2411_03040_gb300 import mgt, synth

H, C, KB = 6.62607015e-34, 299792458.0, 1.380649e-23
SWITCH = 0.35                  # trapezoid below, erf form at or above (the library's default)
COLLIDERS = 1e-4               # collider density out of LTE, as in this repository's Ng experiment


# --------------------------------------------------------------------------
# The cases
# --------------------------------------------------------------------------
def listed():
    return [
        # the smallest solve a user runs: a coarse model iterated to a few ALI
        # steps from LTE, launch and latency bound (the 2,000-point workload)
        dict(name="ali_sphere_2k", op="ali", mesh="sphere", points=2000, levels=5, nside=1, bins=31, iters=4),
        # a survey script: a new model from host arrays, traced, iterated, read
        # back and freed in every pass
        dict(name="oneshot_sphere_5k", op="oneshot", mesh="sphere", points=5000, levels=11, nside=1, bins=31, iters=4),
        # the 64-bit path, run to check the mixed one on a small model
        dict(name="solve64_sphere_2k", op="solve", mesh="sphere", points=2000, levels=5, nside=1, bins=31,
             precision=64),
        # a new velocity snapshot of a hydrodynamics run: fields replaced, rays
        # traced again, one formal solution (few lines: the trace weighs most)
        dict(name="snapshot_sphere_100k", op="snapshot", mesh="sphere", points=100_000, levels=5, nside=2, bins=31),
        # the formal solution of an ALI iteration at the size of the paper's
        # reduced meshes with its 41-level line list (the 100k-point workload)
        dict(name="solve_shell_100k", op="solve", mesh="shell", points=100_000, levels=41, nside=2, bins=50,
             precision=32),
        # rays that do not fit the device: traced 8 pairs at a time inside the
        # formal solution, with a random velocity field (192 rays, 40 bins)
        dict(name="solve_grf_batched_27k", op="solve", mesh="grf", points=27_001, levels=41, nside=4, bins=40,
             precision=32, pairs=8),
        # the statistical equilibrium of every point with 41 levels
        dict(name="equilibrium_shell_100k", op="equilibrium", mesh="shell", points=100_000, levels=41, nside=1, bins=7),
        # many small uneven models per launch: one iteration of a batch
        dict(name="batch_24_small", op="batch", mesh="sphere", models=24, points=500, points_max=5000, bins=31, pick=7),
        # a spectral cube along a held line of sight
        dict(name="image_shell_100k", op="image", mesh="shell", points=100_000, levels=41, px=256, py=256, channels=100),
        # one step of fitting fields to an observed cube: new temperature,
        # density and velocity, the image and its gradient
        dict(name="fit_shell_100k", op="fit", mesh="shell", points=100_000, levels=41, px=128, py=128, channels=64),
        # a model seen from several sides: every view traces its pixel rays
        dict(name="views_shell_100k", op="views", mesh="shell", points=100_000, levels=41, px=128, py=128, channels=32,
             views=2),
        # re-meshing a simulation's point cloud before the transfer
        dict(name="remesh_1m", op="remesh", points=1_000_000, depth=12, r_max=0.4, n_side=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["ali", "oneshot", "solve", "solve64", "solve_batched", "snapshot", "equilibrium", "batch", "image",
                     "fit", "views", "remesh"])
    mesh = rng.choice(["sphere", "shell", "grf"])
    levels = rng.choice([2, 5, 11, 21, 41])
    if op == "remesh":
        return dict(op=op, points=_log(rng, 5000, 1_000_000), depth=rng.choice([4, 8, 12]),
                    r_max=round(rng.uniform(0.2, 0.8), 3), n_side=rng.choice([2, 9, 16]))
    if op == "batch":
        return dict(op=op, mesh="sphere", models=rng.randint(3, 24), points=_log(rng, 200, 1000),
                    points_max=_log(rng, 1500, 5000), bins=rng.choice([9, 16, 31, 40]), pick=rng.randrange(1000))
    if op in ("image", "fit", "views"):
        c = dict(op=op, mesh=mesh, points=_log(rng, 3000, 50_000), levels=levels, px=_log(rng, 8, 200),
                 py=_log(rng, 8, 200), channels=_log(rng, 1, 160))
        if op == "fit":
            c.update(px=min(c["px"], 128), py=min(c["py"], 128), channels=min(c["channels"], 64))
        return dict(c, views=rng.choice([1, 2, 3])) if op == "views" else c
    c = dict(mesh=mesh, points=_log(rng, 700, 40_000), levels=levels, nside=rng.choice([1, 2]), bins=_log(rng, 3, 64))
    if op in ("ali", "oneshot"):
        return dict(c, op=op, points=min(c["points"], 12_000), bins=min(c["bins"], 40), iters=rng.choice([2, 4, 6]))
    if op == "solve64":
        return dict(c, op="solve", points=min(c["points"], 3000), levels=min(levels, 11), nside=1,
                    bins=min(c["bins"], 31), precision=64)
    if op == "solve_batched":
        return dict(c, op="solve", points=min(c["points"], 20_000), nside=2, precision=32, pairs=rng.choice([3, 8]))
    if op == "solve":
        return dict(c, op=op, precision=32)
    return dict(c, op=op)


# --------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------
@functools.lru_cache(maxsize=48)
def _cloud(mesh, n):
    """The point cloud of a kind and size with its graph (model units)."""
    if mesh == "sphere":
        return synth.sphere_model(n, n_levels=2, nside=1, n_quad=1)
    return synth.shell_model(n, n_levels=2, nside=1, n_quad=1)


@functools.lru_cache(maxsize=8)
def _tracer_cloud(n):
    """A cloud on log-spaced radii with a perturbed outflow density, the tracer of the re-meshing."""
    rng = np.random.default_rng(synth.SEED_BASE + n)
    r = np.exp(rng.uniform(0.0, math.log(100.0), n))
    d = rng.normal(size=(n, 3))
    d /= np.linalg.norm(d, axis=1)[:, None]
    rho = 1e16 * np.maximum(r, 0.2) ** -2.0 * (1.0 + 0.3 * np.sin(5.0 * d[:, 0]) * np.cos(3.0 * d[:, 2]))
    return d * r[:, None] * synth.LENGTH_UNIT_M, rho


def _rotation(rng):
    q = rng.normal(size=4)
    w, x, y, z = q / np.linalg.norm(q)
    return np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
                     [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
                     [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]])


def _model(mesh, n, levels, nside, bins, rng):
    base = _cloud(mesh, n)
    rot = _rotation(rng)
    pos, vel = base.pos @ rot.T, base.vel @ rot.T
    if mesh == "grf":
        vel = vel + synth.grf_velocity(pos / synth.LENGTH_UNIT_M, 5e3, 0.05, rng)
    scatter = lambda s: np.exp(s * rng.normal(size=n))
    return synth.Model(f"{mesh}-{n}", pos, vel, base.temp * scatter(0.05), base.vturb2 * scatter(0.1),
                       base.n_coll * COLLIDERS * scatter(0.2), base.n_spec * scatter(0.2), base.nbr_offsets, base.nbrs,
                       base.boundary, synth.healpix_directions(nside), bins, synth.linear_rotor(levels, rng))


def _direction(rng):
    d = rng.normal(size=3)
    return d / np.linalg.norm(d)


def _band(model):
    """Channels across the second line (the first of a two-level molecule)."""
    nu = model.lines.freq_Hz[min(1, model.lines.n_lines - 1)]
    return nu * (1 - 1e-4), nu * (1 + 1e-4)


def _inputs(case, seed):
    """Host inputs of a case, from the seed alone."""
    rng = np.random.default_rng([seed, 2411])
    op = case["op"]
    if op == "remesh":
        # the seed draws the points' order, the axes and the (exact) units, so
        # that the number of boxes belongs to the case
        pos, rho = _tracer_cloud(case["points"])
        order, axes = rng.permutation(case["points"]), rng.permutation(3)
        unit = 2.0 ** rng.integers(-8, 9, 2)
        return dict(pos=np.ascontiguousarray(pos[order][:, axes]) * (unit[0] * rng.choice([-1.0, 1.0], 3)),
                    rho=rho[order] * unit[1])
    if op == "batch":
        specs = synth.batch_specs(case["models"], n_min=case["points"], n_max=case["points_max"], n_quad=case["bins"],
                                  seed=case["pick"])
        return dict(models=[_model(case["mesh"], n, lev, nside, q, rng) for n, lev, nside, q, _ in specs])
    m = _model(case["mesh"], case["points"], case["levels"], case.get("nside", 1), case.get("bins", 7), rng)
    inp = dict(model=m)
    if op == "snapshot":
        inp["vel"] = m.vel * np.exp(0.1 * rng.normal(size=(m.n_points, 1)))
    if op in ("image", "fit", "views"):
        inp["dirs"] = [_direction(rng) for _ in range(case.get("views", 1))]
        inp["band"] = _band(m)
    if op == "fit":
        inp["temp"] = m.temp * np.exp(0.05 * rng.normal(size=m.n_points))
        inp["n_spec"] = m.n_spec * np.exp(0.1 * rng.normal(size=m.n_points))
        inp["vel"] = m.vel * np.exp(0.02 * rng.normal(size=(m.n_points, 1)))
        inp["weight"] = rng.uniform(0.0, 1.0, (case["channels"], case["py"], case["px"])).astype(np.float32)
    return inp


def _device(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a)).to(device="cuda", dtype=dtype)


def _empty(*shape, dtype=torch.float64):
    return torch.empty(shape, dtype=dtype, device="cuda")


def prepare(case, seed):
    mgt.load()
    torch.cuda.set_device(0)
    s = dict(case=case, **_inputs(case, seed))
    op, stream = case["op"], torch.cuda.current_stream()
    if op in ("remesh", "oneshot"):          # calls on host arrays
        return s
    if op == "batch":
        s["handles"] = [mgt.mgt_model_create(m, stream=stream) for m in s["models"]]
        for h in s["handles"]:
            mgt.mgt_trace_rays(h, stream=stream)
        s["batch"] = mgt.mgt_batch_create(s["handles"], stream=stream)
        s["pops"] = [_empty(m.n_points, m.lines.n_levels) for m in s["models"]]
        return s
    m = s["model"]
    n, lines, levels = m.n_points, m.lines.n_lines, m.lines.n_levels
    h = s["h"] = mgt.mgt_model_create(m, stream=stream)
    if op in ("image", "fit", "views"):
        s["out"] = _empty(case.get("views", 1), case["channels"], case["py"], case["px"], dtype=torch.float32)
        if op == "fit":
            for k in ("temp", "n_spec", "vel"):
                s[k] = _device(s[k])
            s["weight"] = _device(s["weight"], torch.float32)
            s["grads"] = _empty(n), _empty(n), _empty(n, 3)
        return s
    if "pairs" in case:
        mgt.mgt_set_solve_opts(h, pairs_per_batch=case["pairs"])
    s["J"], s["L"], s["pops"] = _empty(lines, n), _empty(lines, n), _empty(n, levels)
    if op == "snapshot":
        s["vel"] = _device(s["vel"])
    mgt.mgt_trace_rays(h, stream=stream)
    if op == "equilibrium":
        mgt.mgt_formal_solve(h, mgt.MGT_FP64, want=False, stream=stream)
    return s


# --------------------------------------------------------------------------
# One pass
# --------------------------------------------------------------------------
def _ali(h, iters, stream):
    st = mgt.mgt_ali_solve(h, n_iter=iters, precision=mgt.MGT_FP32_MIXED, ng_mode=mgt.MGT_NG_ADAPTIVE, n_max=8,
                           stream=stream)
    return dict(accepted=st["ng_accepted"], change=st["last_maxrel"])


def run(s):
    case, stream = s["case"], torch.cuda.current_stream()
    op = case["op"]
    if op == "remesh":
        pts, flags = mgt.mgt_remesh(s["pos"], s["rho"], case["r_max"], case["depth"], case["n_side"], stream=stream)
        return dict(points=pts, boundary=flags)
    if op == "oneshot":
        h = mgt.mgt_model_create(s["model"], stream=stream)
        mgt.mgt_trace_rays(h, stream=stream)
        out = _ali(h, case["iters"], stream)
        out["pops"] = mgt.mgt_get_populations(h, stream=stream)
        h.close()
        return out
    if op == "batch":
        for h in s["handles"]:
            mgt.mgt_set_populations(h, None, stream=stream)
        st = mgt.mgt_batch_iterate(s["batch"], 1, mgt.MGT_NG_ADAPTIVE, n_max=8, want_stats=True, stream=stream)
        for h, p in zip(s["handles"], s["pops"]):
            mgt.mgt_get_populations(h, out=p, stream=stream)
        return dict(pops=list(s["pops"]), change=np.array([x["last_maxrel"] for x in st]))
    h = s["h"]
    if op == "ali":
        mgt.mgt_set_populations(h, None, stream=stream)
        out = _ali(h, case["iters"], stream)
        out["pops"] = mgt.mgt_get_populations(h, out=s["pops"], stream=stream)
        return out
    if op == "equilibrium":
        mgt.mgt_stat_equilibrium(h, want=False, stream=stream)
        return mgt.mgt_get_populations(h, out=s["pops"], stream=stream)
    if op in ("solve", "snapshot"):
        if op == "snapshot":
            mgt.mgt_set_point_fields(h, vel=s["vel"], stream=stream)
            mgt.mgt_trace_rays(h, stream=stream)
        p = mgt.MGT_FP64 if case.get("precision") == 64 else mgt.MGT_FP32_MIXED
        return list(mgt.mgt_formal_solve(h, p, s["J"], s["L"], stream=stream))
    px, py, nf = case["px"], case["py"], case["channels"]
    if op == "fit":
        mgt.mgt_set_point_fields(h, s["temp"], s["n_spec"], s["vel"], stream=stream)
    for d, out in zip(s["dirs"], s["out"]):
        mgt.mgt_image(h, d, px, py, nf, *s["band"], out=out, stream=stream)
    if op != "fit":
        return s["out"]
    mgt.mgt_image_adjoint(h, s["dirs"][0], px, py, nf, *s["band"], s["weight"], *s["grads"], stream=stream)
    return [s["out"], *s["grads"]]


# --------------------------------------------------------------------------
# What a pass cannot do without
# --------------------------------------------------------------------------
def _mean_half_ray(mesh, n):
    """Points of a half-ray (measured means: 0.85 N^(1/3) in the shells, about 0.6 N^(1/3) in the sphere)."""
    return (0.6 if mesh == "sphere" else 0.85) * n ** (1.0 / 3.0)


def _solve_work(mesh, n, levels, rays, bins, fp64=False):
    steps = n * rays * _mean_half_ray(mesh, n)
    m = levels - 1
    # per line and step the elimination's 12 flops; per bin and step the segment's coefficients
    return (steps * (32 if fp64 else 16) + n * (2 * m + 2) * (8 if fp64 else 4) + 16 * n * m,
            steps * bins * (12 * m + 40))


def _trace_work(mesh, n, rays):
    steps = n * rays * _mean_half_ray(mesh, n)
    return 16 * steps + 32 * 15.5 * n, steps * 15.5 * 20


def _equilibrium_work(n, levels):
    m = levels - 1
    return n * (16 * levels + 16 * m + 24), n * (2.0 / 3.0 * levels ** 3 + 20 * levels)


def _image_work(mesh, n, levels, px, py, nf):
    # rays that start on the surface end there: about a quarter of two full half-rays each (measured mean)
    seg = px * py * nf * 0.5 * _mean_half_ray(mesh, n)
    return 4.0 * px * py * nf + n * (2 * levels + 8) * 4, 40 * seg


def work(case):
    op = case["op"]
    n, mesh = case.get("points"), case.get("mesh")
    rays = 12 * case.get("nside", 1) ** 2

    def total(*parts):
        return {"bytes": float(sum(b for b, _ in parts)), "flops": float(sum(f for _, f in parts))}

    if op == "remesh":
        levels = min(case["depth"], max(1.0, math.log(n, 8)))
        return total((n * 32.0, n * levels * 16.0))
    if op == "batch":
        parts = []
        for k, lev, nside, q, _ in synth.batch_specs(case["models"], n_min=n, n_max=case["points_max"],
                                                     n_quad=case["bins"], seed=case["pick"]):
            parts += [_solve_work(mesh, k, lev, 12 * nside ** 2, q), _equilibrium_work(k, lev)]
        return total(*parts)
    lev, q = case["levels"], case.get("bins", 7)
    if op in ("image", "fit", "views"):
        b, f = _image_work(mesh, n, lev, case["px"], case["py"], case["channels"])
        v = case.get("views", 1)
        if op == "views":                     # the pixel rays: one row of neighbours per step
            f += case["px"] * case["py"] * 0.5 * _mean_half_ray(mesh, n) * 15.5 * 20
        return total((b * v, f * v)) if op != "fit" else total((b * 2 + 96 * n, f * 4))
    solve = _solve_work(mesh, n, lev, rays, q, case.get("precision") == 64)
    if op in ("ali", "oneshot"):
        parts = [solve, _equilibrium_work(n, lev)] * case["iters"]
        return total(*parts, *([_trace_work(mesh, n, rays)] if op == "oneshot" else []))
    if op == "equilibrium":
        return total(_equilibrium_work(n, lev))
    return total(solve, *([_trace_work(mesh, n, rays)] if op == "snapshot" or "pairs" in case else []))


# --------------------------------------------------------------------------
# The same in plain torch, 64 bits
# --------------------------------------------------------------------------
class _Plain:
    """A model's arrays as 64-bit tensors, with its line tables."""

    def __init__(self, m, temp=None, n_spec=None, vel=None):
        d = lambda a: _device(a)
        self.pos, self.vel = d(m.pos), d(m.vel if vel is None else vel)
        self.temp, self.vt2 = d(m.temp if temp is None else temp), d(m.vturb2)
        self.n_coll, self.n_spec = d(m.n_coll), d(m.n_spec if n_spec is None else n_spec)
        deg = np.diff(m.nbr_offsets)
        pad = np.full((m.n_points, int(deg.max())), -1, np.int64)
        row = np.repeat(np.arange(m.n_points), deg)
        pad[row, np.arange(m.nbrs.size) - np.repeat(m.nbr_offsets[:-1], deg)] = m.nbrs
        self.nbr = torch.as_tensor(pad, device="cuda")
        self.bnd = torch.zeros(m.n_points, dtype=torch.bool, device="cuda")
        self.bnd[torch.as_tensor(m.boundary.astype(np.int64), device="cuda")] = True
        ln = m.lines
        self.E, self.g, self.A, self.nu = d(ln.energy_J), d(ln.g), d(ln.A), d(ln.freq_Hz)
        idx = lambda a: torch.as_tensor(a.astype(np.int64), device="cuda")
        self.up, self.lo, self.cup, self.clo, self.K = idx(ln.up), idx(ln.lo), idx(ln.cup), idx(ln.clo), d(ln.K_ul)
        self.Bul = self.A * C ** 2 / (2 * H * self.nu ** 3)
        self.Blu = self.Bul * self.g[self.up] / self.g[self.lo]
        self.mass, self.T_bg = ln.mol_mass_kg, m.T_bg
        self.w = torch.sqrt(2 * KB * self.temp / self.mass + self.vt2) / C
        self.dirs, self.bins = m.dirs, m.n_quad

    def lte(self):
        b = self.g * torch.exp(-(self.E - self.E[0]) / (KB * self.temp[:, None]))
        return self.n_spec[:, None] * b / b.sum(1, keepdim=True)

    def lines(self, pops):
        """(chi, S) per point and line."""
        a, b = pops[:, self.lo] * self.Blu, pops[:, self.up] * self.Bul
        net = torch.maximum(a - b, 1e-30 * (a + b))
        chi = H * self.nu / (4 * math.pi) * net
        eta = H * self.nu / (4 * math.pi) * pops[:, self.up] * self.A
        return chi, torch.where(chi > 0, eta / torch.where(chi > 0, chi, 1.0), 0.0)

    def planck(self, nu):
        return 2 * H * nu ** 3 / C ** 2 / torch.expm1(H * nu / (KB * self.T_bg))


def _dot(a, b):
    return a[..., 0] * b[..., 0] + a[..., 1] * b[..., 1] + a[..., 2] * b[..., 2]


def _walk(m, start, ref, n, Z):
    """Point lists [T][W] (-1 past the end) of the walks from ``start`` along n through ``ref``."""
    W = start.numel()
    cur, alive, rows = start.clone(), torch.arange(W, device="cuda"), []
    while alive.numel():
        cand = m.nbr[cur[alive]]
        d = m.pos[cand.clamp_min(0)] - ref[alive][:, None, :]
        z = _dot(d, n)
        p = d - z[..., None] * n
        ok = (cand >= 0) & (z > Z[alive][:, None])
        d2 = torch.where(ok, _dot(p, p), math.inf)
        best = d2.amin(1, keepdim=True)
        nxt = torch.where((d2 == best) & ok, cand, 1 << 40).amin(1)
        hit = nxt < 1 << 40
        alive, nxt, cand, z = alive[hit], nxt[hit], cand[hit], z[hit]
        if not alive.numel():
            break
        row = torch.full((W,), -1, dtype=torch.int64, device="cuda")
        row[alive] = nxt
        rows.append(row)
        cur[alive] = nxt
        Z = Z.clone()
        Z[alive] = z.gather(1, (cand == nxt[:, None]).long().argmax(1, keepdim=True))[:, 0]
        alive = alive[~m.bnd[nxt]]
    return torch.stack(rows) if rows else torch.full((0, W), -1, dtype=torch.int64, device="cuda")


def _erf_difference(a, b):
    """erf(b) - erf(a) without cancellation in the tails."""
    flip = a + b < 0
    lo, hi = torch.where(flip, -b, a), torch.where(flip, -a, b)
    return torch.special.erfc(lo) - torch.special.erfc(hi)


def _segment(dx, z0, z1, w0, w1, wbar, shift):
    """c0, c1 with optical depth = (c0 chi0 + c1 chi1) / nu (trapezoid, or the erf form at large shifts)."""
    trap = (shift / wbar).abs() < SWITCH
    t0 = 0.5 * dx * torch.exp(-(z0 / w0) ** 2) / (w0 * math.sqrt(math.pi))
    t1 = 0.5 * dx * torch.exp(-(z1 / w1) ** 2) / (w1 * math.sqrt(math.pi))
    e = 0.25 * dx * _erf_difference(z0 / wbar, z1 / wbar) / torch.where(trap, 1.0, shift)
    return torch.where(trap, t0, e), torch.where(trap, t1, e)


def _half(m, chi, S, rays, n, xw, Ibg):
    """The half-ray's elimination from its far end to the origin: P, Y and the last optical depth."""
    N, M, Q = chi.shape[0], chi.shape[1], xw.shape[1]
    length = (rays >= 0).sum(0)
    order = torch.argsort(length, descending=True)
    length = length[order]
    P = torch.ones((N, M, Q), dtype=torch.float64, device="cuda")
    Y = Ibg[order].clone()
    a = torch.zeros_like(P)
    vo, xw = m.vel[order], xw[order]
    for k in range(rays.shape[0], 0, -1):
        act = int((length >= k).sum())
        o = order[:act]
        f = rays[k - 1][o]
        c = rays[k - 2][o] if k > 1 else o
        bf, bc = ((m.vel[i] - vo[:act]) @ n / C for i in (f, c))
        x, B = xw[:act], 1 + xw[:act]
        wf, wc = m.w[f][:, None], m.w[c][:, None]
        dx = torch.linalg.norm(m.pos[f] - m.pos[c], dim=1)[:, None]
        cf, cc = _segment(dx, x + B * bf[:, None], x + B * bc[:, None], wf, wc, torch.sqrt(0.5 * (wf ** 2 + wc ** 2)),
                          B * (((m.vel[c] - m.vel[f]) @ n) / C)[:, None])
        b = (chi[f] / m.nu)[:, :, None] * cf[:, None, :] + (chi[c] / m.nu)[:, :, None] * cc[:, None, :]
        h = 0.5 * (a[:act] + b)
        Hh = h + P[:act]
        q = 1.0 / (1.0 + b * Hh)
        P[:act] = Hh * q
        Y[:act] = (S[f][:, :, None] * h + Y[:act]) * q
        a[:act] = b
    back = torch.argsort(order)
    return P[back], Y[back], a[back]


def _field(m, pops, rays=None):
    """J-bar and Lambda* [M][N]."""
    chi, S = m.lines(pops)
    x, wq = np.polynomial.hermite.hermgauss(m.bins)
    wq = _device(wq / math.sqrt(math.pi))
    xw = _device(x) * m.w[:, None]
    Ibg = m.planck(m.nu[:, None] * (1 + xw[:, None, :]))
    J, Ls = torch.zeros_like(chi), torch.zeros_like(chi)
    R = m.dirs.shape[0]
    rays = _rays(m) if rays is None else rays
    for r in range(R):
        rb = int(np.argmin(np.linalg.norm(m.dirs + m.dirs[r], axis=1)))
        if rb < r:
            continue
        P0, Y0, a0 = _half(m, chi, S, rays[r], _device(m.dirs[r]), xw, Ibg)
        P1, Y1, a1 = _half(m, chi, S, rays[rb], _device(m.dirs[rb]), xw, Ibg)
        h = 0.5 * (a0 + a1)
        den = h + P0 + P1
        J += 2.0 / R * ((S[:, :, None] * h + Y0 + Y1) / den) @ wq
        Ls += 2.0 / R * (h / den) @ wq
    return J.T.contiguous(), Ls.T.contiguous()


def _rays(m):
    every, zero = torch.arange(m.pos.shape[0], device="cuda"), torch.zeros(m.pos.shape[0], dtype=torch.float64, device="cuda")
    return [_walk(m, every, m.pos, _device(d), zero) for d in m.dirs]


def _equilibrium(m, pops, J, Ls):
    """State reduction of the preconditioned rate equations."""
    N, L = pops.shape
    a, b = pops[:, m.lo] * m.Blu, pops[:, m.up] * m.Bul
    net = torch.maximum(a - b, 1e-30 * (a + b))
    Jeff = J.T - Ls.T * torch.where(net > 0, pops[:, m.up] * m.A / net, 0.0)
    R = torch.zeros((N, L, L), dtype=torch.float64, device="cuda")
    R[:, m.up, m.lo] += torch.clamp_min(m.A * (1 - Ls.T) + m.Bul * Jeff, 0.0)
    R[:, m.lo, m.up] += torch.clamp_min(m.Blu * Jeff, 0.0)
    Cul = m.n_coll[:, None] * m.K
    R[:, m.cup, m.clo] += Cul
    R[:, m.clo, m.cup] += Cul * m.g[m.cup] / m.g[m.clo] * torch.exp(-(m.E[m.cup] - m.E[m.clo]) / (KB * m.temp[:, None]))
    s = torch.zeros((N, L), dtype=torch.float64, device="cuda")
    for n in range(L - 1, 0, -1):
        s[:, n] = R[:, n, :n].sum(1)
        s[:, n] = torch.where(s[:, n] > 0, s[:, n], 1e-300)
        R[:, :n, :n] += R[:, :n, n, None] * (R[:, n, :n] / s[:, n, None])[:, None, :]
    x = torch.zeros((N, L), dtype=torch.float64, device="cuda")
    x[:, 0] = 1.0
    for n in range(1, L):
        x[:, n] = (x[:, :n] * R[:, :n, n]).sum(1) / s[:, n]
    return x / x.sum(1, keepdim=True) * m.n_spec[:, None]


def _change(a, b):
    return float(((a - b).abs() / b.abs())[b != 0].amax())


def _iterate(m, iters):
    """ALI iterations from LTE with the adaptive Ng controller (at most 8 iterates)."""
    rays, pops = _rays(m), m.lte()
    hist, last = [pops / m.n_spec[:, None]], None
    for _ in range(iters):
        new = _equilibrium(m, pops, *_field(m, pops, rays))
        change = _change(new, pops)
        hist.append(new / m.n_spec[:, None])
        pops = new
        if len(hist) == 2:
            last = hist[1]
        if len(hist) < 3:
            continue
        r = torch.stack([(b - a).reshape(-1) for a, b in zip(hist, hist[1:])])
        y = torch.linalg.solve(r @ r.T / (r * r).sum(), torch.ones(len(r), dtype=torch.float64, device="cuda"))
        pred = sum(c * x for c, x in zip(y / y.sum(), hist[1:]))
        if not (_change(pred, last) < change or len(hist) >= 8):
            last = pred
        elif (pred < 0).any():
            hist = hist[-1:]
        else:
            hist, pops = [pred], pred * m.n_spec[:, None]
    return pops


def _pixel_rays(m, n, px, py):
    """Point lists [T][pixels], far end first (-1 past the near end)."""
    ax = min(range(3), key=lambda k: (abs(n[k]), k))
    e1 = np.cross(np.eye(3)[ax], n)
    e1 /= np.linalg.norm(e1)
    e2 = np.cross(n, e1)
    n, e1, e2 = _device(n), _device(e1), _device(e2)
    s1, s2 = _dot(m.pos, e1), _dot(m.pos, e2)
    half = 0.5 * max(float(s1.max() - s1.min()), float(s2.max() - s2.min()))
    grid = lambda s, k: float(s.max() + s.min()) / 2 - half + (torch.arange(k, device="cuda", dtype=torch.float64) + 0.5) * (2 * half / k)
    t2, t1 = torch.meshgrid(grid(s2, py), grid(s1, px), indexing="ij")
    ref = t1.reshape(-1, 1) * e1 + t2.reshape(-1, 1) * e2
    anchor = []
    for r in ref.split(max(1, 20_000_000 // m.pos.shape[0])):
        d = m.pos[None] - r[:, None]
        p = d - _dot(d, n)[..., None] * n
        anchor.append(_dot(p, p).argmin(1))
    anchor = torch.cat(anchor)
    far, near = (_walk(m, anchor, ref, v, _dot(m.pos[anchor] - ref, v)) for v in (-n, n))
    nf, nn = (far >= 0).sum(0), (near >= 0).sum(0)
    out = torch.full((int((nf + nn).max()) + 1, anchor.numel()), -1, dtype=torch.int64, device="cuda")
    q = torch.arange(anchor.numel(), device="cuda")
    out[nf, q] = anchor
    for k in range(far.shape[0]):
        on = far[k] >= 0
        out[nf[on] - 1 - k, q[on]] = far[k][on]
    for k in range(near.shape[0]):
        on = near[k] >= 0
        out[nf[on] + 1 + k, q[on]] = near[k][on]
    return out


def _cube(m, chi, S, w, vel, n, rays, nf, band):
    """Intensities [channels][pixels], the rays longest first (and their order)."""
    nu = torch.linspace(*band, nf, dtype=torch.float64, device="cuda") if nf > 1 else _device([band[0]])
    line = (nu[:, None] - m.nu).abs().argmin(1)
    nl, r = m.nu[line], nu / m.nu[line]
    length = (rays >= 0).sum(0)
    order = torch.argsort(length, descending=True)
    length, rays = length[order], rays[:, order]
    beta = vel @ _device(n) / C
    I = m.planck(nu).expand(rays.shape[1], nf)
    for d in range(rays.shape[0] - 1):
        act = int((length > d + 1).sum())
        a, b = rays[d][:act], rays[d + 1][:act]
        dx = torch.linalg.norm(m.pos[b] - m.pos[a], dim=1)[:, None]
        wa, wb = w[a][:, None], w[b][:, None]
        za, zb = ((r * (1 - beta[i][:, None])) - 1 for i in (a, b))
        ca, cb = _segment(dx, za, zb, wa, wb, torch.sqrt(0.5 * (wa ** 2 + wb ** 2)), r * (beta[a] - beta[b])[:, None])
        t = (ca * chi[a][:, line] + cb * chi[b][:, line]) / nl
        E, small = torch.exp(-t), t < 1e-3
        ts = torch.where(small, 1.0, t)
        g = torch.where(small, 1 - t / 2 + t ** 2 / 6 - t ** 3 / 24 + t ** 4 / 120, (1 - torch.exp(-ts)) / ts)
        new = E * I[:act] + (g - E) * S[a][:, line] + (1 - g) * S[b][:, line]
        I = torch.cat([new, I[act:]])
    return I.T, order


def _image(m, pops, case, d, band, weight=None):
    rays = _pixel_rays(m, d, case["px"], case["py"])
    chi, S = m.lines(pops)
    shape = (case["channels"], case["py"], case["px"])
    if weight is None:
        I, order = _cube(m, chi, S, m.w, m.vel, d, rays, case["channels"], band)
        return I[:, torch.argsort(order)].reshape(shape)
    logT, logn = (torch.zeros_like(m.temp, requires_grad=True) for _ in range(2))
    vel = m.vel.clone().requires_grad_()
    image, part = [], max(1, 1_000_000 // case["channels"])
    for q in range(0, rays.shape[1], part):           # the pixels in parts: a part's graph fits the memory
        w = torch.sqrt(2 * KB * m.temp * torch.exp(logT) / m.mass + m.vt2) / C
        I, order = _cube(m, chi * torch.exp(logn)[:, None], S, w, vel, d, rays[:, q:q + part], case["channels"], band)
        I = I[:, torch.argsort(order)]
        (I * weight.reshape(case["channels"], -1)[:, q:q + part]).sum().backward()
        image.append(I.detach())
    return [torch.cat(image, 1).reshape(shape)[None], logT.grad, logn.grad, vel.grad]


def _remesh(pos, rho, r_max, depth, n_side):
    perm, start = np.arange(len(rho)), np.array([0])
    leaves, root = [], None
    for level in range(depth + 1):
        p, t = pos[perm], rho[perm]
        lo, hi = np.minimum.reduceat(p, start), np.maximum.reduceat(p, start)
        tmin, tmax = np.minimum.reduceat(t, start), np.maximum.reduceat(t, start)
        root = (lo[0], hi[0]) if root is None else root
        mid = (lo + hi) * 0.5
        split = (2.0 * ((tmax - tmin) / (tmax + tmin)) > r_max) & (level < depth)
        leaves.append(mid[~split])
        if not split.any():
            break
        box = np.repeat(np.arange(len(start)), np.diff(np.append(start, len(perm))))
        keep = split[box]
        box, perm, p = box[keep], perm[keep], p[keep]
        key = box * 8 + ((p >= mid[box]) @ np.array([1, 2, 4]))
        order = np.argsort(key, kind="stable")
        perm, key = perm[order], key[order]
        start = np.concatenate([[0], np.nonzero(np.diff(key))[0] + 1])
    k = np.arange(n_side)
    ijk = np.stack(np.meshgrid(k, k, k, indexing="ij"), -1).reshape(-1, 3)
    ijk = ijk[((ijk == 0) | (ijk == n_side - 1)).any(1)]
    leaves = np.concatenate(leaves)
    pts = np.concatenate([leaves, root[0] + ijk / (n_side - 1) * (root[1] - root[0])])
    return dict(points=pts, boundary=(np.arange(len(pts)) >= len(leaves)).astype(np.uint8))


def exact(case, seed):
    op = case["op"]
    if op in ("solve", "snapshot", "ali", "oneshot"):
        times = case.get("iters", 1)
        line_steps = (case["points"] * 12 * case["nside"] ** 2 * _mean_half_ray(case["mesh"], case["points"]) *
                      case["bins"] * (case["levels"] - 1 + 4))
        if line_steps * times > 6e10:          # over the time that a reference may take
            return None
    torch.cuda.set_device(0)
    s = _inputs(case, seed)
    if op == "remesh":
        return _remesh(s["pos"], s["rho"], case["r_max"], case["depth"], case["n_side"])
    if op == "batch":
        return dict(pops=[_iterate(_Plain(m), 1) for m in s["models"]], change=None)
    fields = {k: s[k] for k in ("temp", "n_spec", "vel") if k in s}
    m = _Plain(s["model"], **fields)
    if op in ("ali", "oneshot"):
        return dict(accepted=None, change=None, pops=_iterate(m, case["iters"]))
    # populations are held as fractions of the species density from the model's own LTE
    own = _Plain(s["model"])
    pops = own.lte() / own.n_spec[:, None] * m.n_spec[:, None]
    if op in ("solve", "snapshot"):
        return list(_field(m, pops))
    if op == "equilibrium":
        return _equilibrium(m, pops, *_field(m, pops))
    if op == "fit":
        return _image(m, pops, case, s["dirs"][0], s["band"], _device(s["weight"]))
    return torch.stack([_image(m, pops, case, d, s["band"]) for d in s["dirs"]])
