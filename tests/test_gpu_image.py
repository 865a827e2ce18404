"""Synthetic image (mgt_image) and its adjoint against the CPU oracle, through the C-ABI.

Tolerances: pixel rays bit-exact (anchors and point lists); image 1e-4
relative per pixel and channel (FP32 path); adjoint gradients against the
oracle's FP64 gradient (a reverse sweep of its image solve) element by element
on 64 points, within 2e-3 relative plus 2e-4 of the field's largest sampled
gradient; against central differences of the GPU image on 64 points (h = 1e-4
in log T and log n_spec, 1 m/s in velocity; FP32 images differenced pixel by
pixel, unaffected pixels cancel exactly) within 2e-2 of the largest, leaving
out only (point, field) pairs whose step moves a segment across the
trapezoid / erf switch (found from the oracle's branch map).
"""
import numpy as np
import pytest

import oracle as O
from paper_2411_03040_gb300 import synth

pytestmark = pytest.mark.gpu

DIR = np.array([0.3, -0.5, 0.8]) / np.linalg.norm([0.3, -0.5, 0.8])
# adjoint (FP32) against the oracle's FP64 gradient: relative, with an absolute
# floor of the field's largest sampled gradient for entries that are sums of
# contributions of both signs
RTOL_ADJ, ATOL_ADJ = 2e-3, 2e-4


@pytest.fixture(scope="module")
def mgt():
    from paper_2411_03040_gb300 import build, mgt as binding
    build.build()
    binding.load()
    return binding


def _band(model, line=0, halfwidth=4e-5):
    nu0 = model.lines.freq_Hz[line]
    return nu0 * (1 - halfwidth), nu0 * (1 + halfwidth)


def _pops(model):
    return O.lte_populations(model.temp, model.n_spec, model.lines.energy_J, model.lines.g)


@pytest.mark.parametrize("case", ["sphere", "shell-grf", "lattice"])
def test_pixel_rays_bit_exact(mgt, case):
    if case == "sphere":
        m, d, npx, npy = synth.config_model(1, n_points=800), DIR, 12, 10
    elif case == "shell-grf":
        m, d, npx, npy = synth.shell_model(3000, 3, 1, 5, grf_sigma=5e3, seed=8, name="grf"), DIR, 16, 16
    else:
        m, d, npx, npy = synth.lattice_model(n_side=7), np.array([0.0, 0.0, 1.0]), 7, 7
    h = mgt.mgt_model_create(m)
    anchor, off, pts = mgt.mgt_image_rays(h, d, npx, npy)
    r = O.image_rays(m, d, npx, npy)
    assert np.array_equal(anchor, r.anchor)
    assert np.array_equal(off, r.off)
    assert np.array_equal(pts, r.pts)


@pytest.mark.parametrize("case", ["sphere", "shell-grf"])
def test_image_matches_oracle(mgt, case):
    if case == "sphere":
        m = synth.config_model(1, n_points=800)
    else:
        m = synth.shell_model(3000, 4, 1, 5, grf_sigma=5e3, seed=8, name="grf")
    lo, hi = _band(m)
    h = mgt.mgt_model_create(m)
    img = mgt.mgt_image(h, DIR, 12, 10, 21, lo, hi)
    ref, _ = O.image(m, _pops(m), DIR, 12, 10, 21, lo, hi)
    err = np.max(np.abs(img - ref) / np.abs(ref))
    assert err < 1e-4, err
    # a second line, and device output
    import torch
    lo2, hi2 = _band(m, line=2)
    out = torch.zeros((7, 10, 12), dtype=torch.float32, device="cuda")
    mgt.mgt_image(h, DIR, 12, 10, 7, lo2, hi2, out=out)
    ref2, _ = O.image(m, _pops(m), DIR, 12, 10, 7, lo2, hi2)
    assert np.max(np.abs(out.cpu().numpy() - ref2) / np.abs(ref2)) < 1e-4


@pytest.mark.parametrize("npx,npy,nfreq,band", [(1, 1, 1, "centre"), (1, 9, 300, "line"), (5, 1, 2, "wings")],
                         ids=["1x1-one-channel", "column-300-channels", "row-two-wing-channels"])
def test_image_degenerate_sizes(mgt, npx, npy, nfreq, band):
    # one pixel and one channel at the line centre (fmin = fmax); a one-pixel
    # column of 300 channels (two trips of a 256-thread block over the
    # channels); a one-pixel row of two channels far in the wings of the first
    # two lines, where the image is the background
    m = synth.config_model(1, n_points=800)
    nu0, nu1 = m.lines.freq_Hz[0], m.lines.freq_Hz[1]
    lo, hi = {"centre": (nu0, nu0), "line": _band(m), "wings": (0.9 * nu0, 1.1 * nu1)}[band]
    h = mgt.mgt_model_create(m)
    img = mgt.mgt_image(h, DIR, npx, npy, nfreq, lo, hi)
    ref, _ = O.image(m, _pops(m), DIR, npx, npy, nfreq, lo, hi)
    assert img.shape == ref.shape == (nfreq, npy, npx)
    err = np.max(np.abs(img - ref) / np.abs(ref))
    assert err < 1e-4, err
    if band == "wings":
        bg = np.array([O.planck(f, m.T_bg) for f in (lo, hi)])
        assert np.max(np.abs(ref[:, 0, :] / bg[:, None] - 1)) < 1e-6
    if band == "centre":
        # the adjoint of the one-pixel, one-channel image: every point of its
        # ray against the oracle's FP64 gradient, zero off the ray
        w = np.ones((1, 1, 1), np.float32)
        grads = mgt.mgt_image_adjoint(h, DIR, 1, 1, 1, lo, hi, w)
        rays = O.image_rays(m, DIR, 1, 1)
        refs = O.image_adjoint(m, _pops(m), DIR, 1, 1, 1, lo, hi, w.astype(np.float64), rays=rays)
        on = np.unique(rays.pts)
        off = np.setdiff1d(np.arange(m.n_points), on)
        for key, g, r in zip("Tnv", grads, refs):
            assert np.all(g[off] == 0) and np.all(r[off] == 0), key
            scale = np.max(np.abs(r[on]))
            assert scale > 0, key
            assert np.all(np.abs(g[on] - r[on]) <= RTOL_ADJ * np.abs(r[on]) + ATOL_ADJ * scale), key


def test_adjoint_matches_oracle_gradient(mgt):
    # element by element against the oracle's FP64 reverse sweep, on 64 random
    # points of the pixel rays, all three fields (the velocity gradient lies
    # along the line of sight on both sides)
    m = synth.config_model(1, n_points=600)
    npx, npy, nfreq = 12, 12, 15
    lo, hi = _band(m)
    rng = np.random.default_rng(3)
    w = rng.uniform(0.0, 1.0, size=(nfreq, npy, npx))
    h = mgt.mgt_model_create(m)
    gT, gn, gv = mgt.mgt_image_adjoint(h, DIR, npx, npy, nfreq, lo, hi, w.astype(np.float32))
    rays = O.image_rays(m, DIR, npx, npy)
    rT, rn, rv = O.image_adjoint(m, _pops(m), DIR, npx, npy, nfreq, lo, hi, w.astype(np.float32).astype(np.float64),
                                 rays=rays)
    pick = rng.choice(np.unique(rays.pts), size=64, replace=False)
    for key, g, ref in (("T", gT, rT), ("n", gn, rn), ("v", gv, rv)):
        g, ref = g[pick], ref[pick]
        scale = np.max(np.abs(ref))
        assert scale > 0
        err = np.abs(g - ref)
        assert np.all(err <= RTOL_ADJ * np.abs(ref) + ATOL_ADJ * scale), (key, np.max(err / (np.abs(ref) + scale)))


def test_adjoint_matches_gpu_finite_differences_and_autograd(mgt):
    import torch
    m = synth.config_model(1, n_points=500)
    npx, npy, nfreq = 16, 16, 20
    lo, hi = _band(m)
    rng = np.random.default_rng(5)
    w = rng.uniform(0.0, 1.0, size=(nfreq, npy, npx))
    h = mgt.mgt_model_create(m)
    gT, gn, gv = mgt.mgt_image_adjoint(h, DIR, npx, npy, nfreq, lo, hi, w.astype(np.float32))
    _, _, pts = mgt.mgt_image_rays(h, DIR, npx, npy)
    pick = rng.choice(np.unique(pts), size=64, replace=False)
    hstep = 1e-4

    def loss(T, n, v):
        mgt.mgt_set_point_fields(h, T, n, v)
        img = mgt.mgt_image(h, DIR, npx, npy, nfreq, lo, hi)
        return img.astype(np.float64)

    T0, n0, v0 = m.temp.copy(), m.n_spec.copy(), m.vel.copy()
    rays = O.image_rays(m, DIR, npx, npy)
    base_br = O.image_branches(m, DIR, nfreq, lo, hi, rays)
    res = []
    flips = 0
    for c in pick:
        for key, g in (("T", gT[c]), ("n", gn[c]), ("v", gv[c] @ DIR)):
            imgs, same = [], True
            for sgn in (1, -1):
                T, n, v = T0.copy(), n0.copy(), v0.copy()
                if key == "T":
                    T[c] *= np.exp(sgn * hstep)
                elif key == "n":
                    n[c] *= np.exp(sgn * hstep)
                else:
                    v[c] = v[c] + sgn * 1.0 * DIR                  # 1 m/s
                imgs.append(loss(T, n, v))
                mm = synth.Model(m.name, m.pos, v, T, m.vturb2, m.n_coll, n, m.nbr_offsets, m.nbrs, m.boundary,
                                 m.dirs, m.n_quad, m.lines, m.T_bg)
                same = same and np.array_equal(O.image_branches(mm, DIR, nfreq, lo, hi, rays), base_br)
            step = hstep if key != "v" else 1.0
            fdv = float(np.sum(w * (imgs[0] - imgs[1]))) / (2 * step)
            if same:
                res.append((key, g, fdv))
            else:
                flips += 1
    mgt.mgt_set_point_fields(h, T0, n0, v0)
    # A finite step that moves a segment across the trapezoid / erf switch
    # makes the image jump (the two forms differ slightly at the threshold), so
    # the difference quotient means nothing there: such (point, field) pairs,
    # found from the oracle's branch map of the perturbed fields, are left out.
    assert flips <= 8, flips
    for key in ("T", "n", "v"):
        g = np.array([b[1] for b in res if b[0] == key])
        f = np.array([b[2] for b in res if b[0] == key])
        assert g.size >= 56
        assert np.all(np.abs(g - f) < 2e-2 * np.max(np.abs(f))), (key, np.max(np.abs(g - f)) / np.max(np.abs(f)))
    # the autograd.Function gives the same gradients as the direct adjoint call
    from paper_2411_03040_gb300.autograd import ImageFunction
    lt = torch.tensor(np.log(T0), device="cuda", requires_grad=True)
    ln = torch.tensor(np.log(n0), device="cuda", requires_grad=True)
    vv = torch.tensor(v0, device="cuda", requires_grad=True)
    img = ImageFunction.apply(lt, ln, vv, h, DIR, npx, npy, nfreq, lo, hi)
    (img.double() * torch.tensor(w, device="cuda")).sum().backward()
    assert np.allclose(lt.grad.cpu().numpy(), gT, rtol=1e-9, atol=0)
    assert np.allclose(ln.grad.cpu().numpy(), gn, rtol=1e-9, atol=0)
    assert np.allclose(vv.grad.cpu().numpy(), gv, rtol=1e-9, atol=0)


@pytest.mark.parametrize("n,npx,npy,shape", [(1, 3, 2, "ball"), (7, 5, 5, "ball"), (400, 33, 7, "ball"),
                                             (400, 9, 9, "line"), (400, 9, 9, "plane"), (5000, 40, 40, "clumps"),
                                             (5000, 12, 12, "far")])
def test_pixel_rays_of_awkward_clouds(mgt, n, npx, npy, shape):
    # anchors found through the search grid: one cell only, every projection on
    # one place or on a line, empty corners, thousands of points in one cell
    # and coincident points (ties), a cloud far from the origin (bounds wider
    # than a cell).  Rays are decided by FP64 predicates: equality
    rng = np.random.default_rng(n + npx)
    pos = rng.normal(size=(n, 3))
    d = np.array([0.0, 0.0, 1.0])
    if shape == "line":
        pos[:, :2] = 0.25
    elif shape == "plane":
        pos[:, 0] = 0.0
    elif shape == "clumps":
        pos[: n // 2] = np.round(pos[: n // 2] * 1e-3, 4)
        pos[::50] *= 30.0
        d = DIR
    elif shape == "far":
        pos = pos * 1e-4 + np.array([1.0, -2.0, 0.5])
        d = DIR
    nb = [rng.choice(n, size=min(n, 8), replace=False) for _ in range(n)]
    off = np.concatenate([[0], np.cumsum([len(v) for v in nb])]).astype(np.int64)
    m = synth.Model("cloud", pos * 1e11, np.zeros((n, 3)), np.full(n, 50.0), np.full(n, 1e4), np.full(n, 1e10),
                    np.full(n, 1e5), off, np.concatenate([np.sort(v) for v in nb]).astype(np.int32),
                    np.arange(0, n, 10, dtype=np.int32), synth.healpix_directions(1), 3, synth.linear_rotor(3, rng))
    h = mgt.mgt_model_create(m)
    for direction in (d, -d):                  # the second view reuses the first one's buffers
        anchor, roff, pts = mgt.mgt_image_rays(h, direction, npx, npy)
        r = O.image_rays(m, direction, npx, npy)
        assert np.array_equal(anchor, r.anchor)
        assert np.array_equal(roff, r.off) and np.array_equal(pts, r.pts)


def test_pixel_rays_longer_than_their_slots(mgt):
    # a chain along the line of sight: half-rays of up to 1,500 points, beyond
    # the scratch slot (8 n^(1/3) + 16), are walked again into their place
    n = 1500
    x = np.linspace(-1, 1, n)
    pos = np.stack([0.05 * x ** 2, 0.01 * np.sin(3 * x), x], axis=1)
    nb = [[j for j in (i - 1, i + 1) if 0 <= j < n] for i in range(n)]
    off = np.concatenate([[0], np.cumsum([len(v) for v in nb])]).astype(np.int64)
    rng = np.random.default_rng(3)
    m = synth.Model("chain", pos * 1e11, np.zeros((n, 3)), np.full(n, 50.0), np.full(n, 1e4), np.full(n, 1e10),
                    np.full(n, 1e5), off, np.concatenate(nb).astype(np.int32), np.array([0, n - 1], np.int32),
                    synth.healpix_directions(1), 3, synth.linear_rotor(3, rng))
    d = np.array([0.0, 0.0, 1.0])
    h = mgt.mgt_model_create(m)
    anchor, roff, pts = mgt.mgt_image_rays(h, d, 4, 3)
    r = O.image_rays(m, d, 4, 3)
    assert np.max(np.diff(roff)) > 1000
    assert np.array_equal(anchor, r.anchor) and np.array_equal(roff, r.off) and np.array_equal(pts, r.pts)


@pytest.mark.parametrize("nfreq", [32, 33, 63, 65, 514])
def test_channel_counts_around_the_pairs(mgt, nfreq):
    # one channel per thread up to 32 channels, two neighbours per thread above
    # (an odd last one, more than one trip of 256 pairs), over a band of three
    # lines, so that some pairs see different lines; tolerance of the images
    m = synth.shell_model(3000, 4, 1, 5, grf_sigma=2e3, seed=8, name="grf")
    nu = m.lines.freq_Hz
    lo, hi = 0.9999 * nu[0], 1.0001 * nu[2]
    h = mgt.mgt_model_create(m)
    for a, b in ((lo, hi), _band(m, line=1)):
        img = mgt.mgt_image(h, DIR, 5, 4, nfreq, a, b)
        ref, _ = O.image(m, _pops(m), DIR, 5, 4, nfreq, a, b)
        assert np.max(np.abs(img - ref) / np.abs(ref)) < 1e-4


@pytest.mark.parametrize("nfreq", [64, 96, 97, 128, 129, 160, 161, 257])
def test_channel_counts_where_pairs_begin_and_end(mgt, nfreq):
    # two channels per thread where that saves enough warps (33 to 64 channels,
    # 97 to 128, from 161), one per thread elsewhere; one line and a band of
    # three; tolerance of the images
    m = synth.shell_model(1500, 4, 1, 5, grf_sigma=2e3, seed=8, name="grf")
    nu = m.lines.freq_Hz
    h = mgt.mgt_model_create(m)
    for a, b in ((0.9999 * nu[0], 1.0001 * nu[2]), _band(m, line=1)):
        img = mgt.mgt_image(h, DIR, 3, 4, nfreq, a, b)
        ref, _ = O.image(m, _pops(m), DIR, 3, 4, nfreq, a, b)
        assert np.max(np.abs(img - ref) / np.abs(ref)) < 1e-4


def _bare_cloud(pos, rng):
    """Points with random neighbours and plain fields, for the pixel rays alone."""
    n = pos.shape[0]
    nb = [rng.choice(n, size=8, replace=False) for _ in range(n)]
    return synth.Model("cloud", pos, np.zeros((n, 3)), np.full(n, 50.0), np.full(n, 1e4), np.full(n, 1e10),
                       np.full(n, 1e5), 8 * np.arange(n + 1, dtype=np.int64),
                       np.concatenate([np.sort(v) for v in nb]).astype(np.int32), np.arange(0, n, 10, dtype=np.int32),
                       synth.healpix_directions(1), 3, synth.linear_rotor(3, rng))


def test_anchors_among_points_closer_than_float_pairs_resolve(mgt):
    # around every pixel's reference point eight points at 1e-11 of the model's
    # extent from the pixel line, whose distances differ by less than float
    # hi + lo positions resolve: FP64 decides, equality
    rng = np.random.default_rng(17)
    npx, npy = 12, 10
    pos = rng.uniform(-1, 1, size=(200, 3)) * 1e11
    r = O.image_rays(_bare_cloud(pos, rng), DIR, npx, npy)
    ang = rng.uniform(0, 2 * np.pi, (npx * npy, 8))
    rad = 1.0 + rng.uniform(0.0, 4e-4, ang.shape)                     # m: 4e-15 of 1e11 m
    off = rad[..., None] * (np.cos(ang)[..., None] * r.e1 + np.sin(ang)[..., None] * r.e2)
    near = (r.ref[:, None, :] + off).reshape(-1, 3)
    inside = np.all(np.abs(near) < 0.9e11, axis=1)                   # the frame stays the cloud's
    assert inside.sum() > 200
    m = _bare_cloud(np.concatenate([pos, near[inside]]), rng)
    ref = O.image_rays(m, DIR, npx, npy)
    assert np.array_equal(ref.ref, r.ref) and (ref.anchor >= 200).sum() > 40
    anchor, _, _ = mgt.mgt_image_rays(mgt.mgt_model_create(m), DIR, npx, npy)
    assert np.array_equal(anchor, ref.anchor)


def test_anchors_of_a_small_cloud_far_away_with_a_rounded_direction(mgt):
    # a direction as far from unit length as the call accepts shifts the pixels
    # against the projections by 1e-12 of their distance from the plane's
    # origin: here by about a cell of the search grid (points in the plane of
    # the reference points, 1.2 from its origin).  FP64 decides, equality
    rng = np.random.default_rng(23)
    d = np.array([-0.576, 0.578, 0.578]) / np.linalg.norm([-0.576, 0.578, 0.578])
    e2 = np.array([1.0, 0.0, 0.0]) - d[0] * d
    e2 /= np.linalg.norm(e2)
    uv = rng.uniform(-3e-11, 3e-11, size=(5000, 2))
    m = _bare_cloud((1.2 * e2 + uv[:, :1] * np.cross(d, e2) + uv[:, 1:] * e2) * 2.0 ** 37, rng)
    h = mgt.mgt_model_create(m)
    for scale in (1.0 - 4.9e-13, 1.0 + 4.9e-13):
        anchor, _, _ = mgt.mgt_image_rays(h, d * scale, 80, 80)
        assert np.array_equal(anchor, O.image_rays(m, d * scale, 80, 80).anchor)


def test_held_view_read_on_two_streams(mgt):
    # the kept pixel rays are read on a second stream while the first one asks
    # for another view: its rays must not be written over those being read.
    # The images of one stream alone, bit for bit
    import torch
    m = synth.sphere_model(3000, 5, 1, 5, seed=12)
    lo, hi = _band(m)
    views = [DIR, -DIR, np.array([0.0, 0.0, 1.0])]
    px, nf = 96, 200
    h = mgt.mgt_model_create(m)
    out = [torch.empty((nf, px, px), dtype=torch.float32, device="cuda") for _ in range(6)]
    for v, o in zip(views, out):
        mgt.mgt_image(h, v, px, px, nf, lo, hi, out=o)
    torch.cuda.synchronize()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(3):
        for k in (0, 1):
            for o in out[3:]:
                o.zero_()
            torch.cuda.synchronize()
            mgt.mgt_image(h, views[k], px, px, nf, lo, hi, out=out[3], stream=s1)
            mgt.mgt_image(h, views[k], px, px, nf, lo, hi, out=out[4], stream=s2)
            mgt.mgt_image(h, views[k + 1], px, px, nf, lo, hi, out=out[5], stream=s1)
            torch.cuda.synchronize()
            assert torch.equal(out[3], out[k]) and torch.equal(out[4], out[k]) and torch.equal(out[5], out[k + 1])
