"""The ray walk on rows of awkward lengths, through the C-ABI against the oracle.

Point lists are decided by FP64 predicates: equality, no tolerance.
"""
import numpy as np
import pytest

import oracle as O
from paper_2411_03040_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mgt():
    from paper_2411_03040_gb300 import build, mgt as binding
    build.build()
    binding.load()
    return binding


def _model(pos, nbrs, boundary, rng):
    n = len(pos)
    off = np.concatenate([[0], np.cumsum([len(v) for v in nbrs])]).astype(np.int64)
    flat = np.concatenate([np.sort(np.asarray(v, np.int32)) for v in nbrs]) if off[-1] else np.zeros(0, np.int32)
    return synth.Model("graph", pos * 1e11, rng.normal(size=(n, 3)) * 1e3, np.full(n, 50.0), np.full(n, 1e4),
                       np.full(n, 1e10), np.full(n, 1e5), off, flat.astype(np.int32), np.asarray(boundary, np.int32),
                       synth.healpix_directions(1), 3, synth.linear_rotor(3, rng))


@pytest.mark.parametrize("n,degrees", [(1, [0]), (9, [0, 1]), (40, [3, 4, 5]), (300, [0, 1, 2, 3, 4, 5, 7, 8, 9]),
                                       (200, [31, 32, 33, 40]), (4100, [0, 1, 2, 3, 4, 5, 7, 8, 9, 17])], ids=str)
def test_rows_around_chunk_edges(mgt, n, degrees):
    # rows with no, one and a few more or less than whole chunks of entries,
    # rows above one warp's lanes, and fewer walks than the last warp holds; the
    # largest (49,200 walks) runs 4 lanes per walk, the others 16
    rng = np.random.default_rng(n)
    pos = rng.uniform(-1, 1, size=(n, 3))
    pos[n // 2:] = np.round(pos[n // 2:] * 4) / 4          # coincident and collinear points: ties and undecided steps
    nbrs = [rng.choice(n, size=min(n, degrees[i % len(degrees)]), replace=False) for i in range(n)]
    m = _model(pos, nbrs, rng.choice(n, size=max(1, n // 10), replace=False), rng)
    h = mgt.mgt_model_create(m)
    st = mgt.mgt_trace_rays(h)
    off, idx = mgt.mgt_get_rays(h)
    r = O.trace(m)
    assert np.array_equal(off, r.off) and np.array_equal(idx, r.idx)
    assert st["n_stalls"] == r.stalls and st["total_steps"] == r.off[-1]


@pytest.mark.parametrize("jitter", [0.0, 1e-15, 1e-13, 1e-10, 1e-8, 1e-7, 1e-6, 1e-4])
@pytest.mark.parametrize("side,shift", [(12, 0.0), (16, 0.0), (16, 40.0)])
def test_near_ties_at_every_scale(mgt, side, shift, jitter):
    # a lattice disturbed by less or more than the filter's error bounds: along
    # the axes and the diagonals of the 12 directions candidates tie up to the
    # jitter, in projection and in distance; with the shift the coordinates are
    # large against the spacing; 12 a side runs 16 lanes per walk, 16 a side 4
    rng = np.random.default_rng(7)
    g = np.arange(side)
    pos = np.stack(np.meshgrid(g, g, g, indexing="ij"), axis=-1).reshape(-1, 3).astype(float)
    nbrs = []
    for i, p in enumerate(pos):
        d = np.abs(pos - p).max(axis=1)
        nbrs.append(np.flatnonzero((d <= 1) & (np.arange(len(pos)) != i)))
    edge = np.flatnonzero((pos.min(axis=1) == 0) | (pos.max(axis=1) == side - 1))
    m = _model(pos + shift + jitter * rng.normal(size=pos.shape), nbrs, edge, rng)
    h = mgt.mgt_model_create(m)
    mgt.mgt_trace_rays(h)
    off, idx = mgt.mgt_get_rays(h)
    r = O.trace(m)
    assert np.array_equal(off, r.off) and np.array_equal(idx, r.idx)


@pytest.mark.parametrize("n", [300, 700])
def test_walks_longer_than_the_first_guess(mgt, n):
    # a bent chain: half-rays up to n - 1 points, beyond the first trace's slot
    # (four times 4 n^(1/3) + 16), so they are walked again into their final place; the
    # records are checked through the formal solution, traced twice
    rng = np.random.default_rng(n)
    x = np.linspace(-1, 1, n)
    pos = np.stack([x, 0.05 * x ** 2, 0.01 * np.sin(3 * x)], axis=1)
    nbrs = [[j for j in (i - 1, i + 1) if 0 <= j < n] for i in range(n)]
    m = _model(pos, nbrs, [0, n - 1], rng)
    h = mgt.mgt_model_create(m)
    st = mgt.mgt_trace_rays(h)
    r = O.trace(m)
    off, idx = mgt.mgt_get_rays(h)
    assert st["max_half_ray"] > 4 * (4 * n ** (1 / 3) + 32)
    assert np.array_equal(off, r.off) and np.array_equal(idx, r.idx)
    first = mgt.mgt_formal_solve(h)
    mgt.mgt_trace_rays(h)                                  # the slot now holds every walk
    again = mgt.mgt_formal_solve(h)
    assert all(np.array_equal(a, b) for a, b in zip(first, again))
