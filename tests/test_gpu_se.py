"""Statistical equilibrium at the edges of its lane and point groups, through
the C-ABI against the oracle on the model's own J-bar and Lambda*.

Tolerance 1e-8 relative, element by element, as in the parity tests: the state
reduction keeps populations to about 2 L^3 rounding units (6e-11 at 64 levels),
and the preconditioned rates lose digits where J-bar - Lambda* S cancels.
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


# lanes per point change above 16 and 32 levels; point counts leave the last
# warp with one, some and all of its points
@pytest.mark.parametrize("levels,n", [(2, 31), (3, 64), (15, 33), (16, 40), (17, 41), (31, 37), (32, 30), (33, 31),
                                      (63, 29), (64, 32)])
@pytest.mark.parametrize("batched", [False, True])
def test_level_and_point_edges(mgt, levels, n, batched):
    m = synth.sphere_model(n, levels, 1, 3, seed=50 + levels)
    m.n_coll = m.n_coll * 1e-4
    h = mgt.mgt_model_create(m)
    mgt.mgt_trace_rays(h)
    if batched:
        other = synth.sphere_model(60, 5, 1, 3, seed=7)
        ho = mgt.mgt_model_create(other)
        mgt.mgt_trace_rays(ho)
        b = mgt.mgt_batch_create([ho, h])
        mgt.mgt_batch_formal_solve(b)
        mgt.mgt_batch_stat_equilibrium(b)
        got = mgt.mgt_get_populations(h)
    else:
        mgt.mgt_formal_solve(h, want=False)
        got = mgt.mgt_stat_equilibrium(h)
    J, L = mgt.mgt_get_jbar(h)
    p0 = O.lte_populations(m.temp, m.n_spec, m.lines.energy_J, m.lines.g)
    ref = O.stat_equilibrium(p0, J.T, L.T, m.temp, m.n_coll, m.n_spec, m.lines)
    assert np.max(np.abs(got - ref) / np.abs(ref)) < 1e-8
    # the previous populations are kept for the change that Ng reports
    _, change = mgt.mgt_ng_accelerate(h)
    assert change == pytest.approx(np.max(np.abs(got - p0) / p0), rel=1e-9)


# (levels, points): every number of lanes per point, whose choice depends on both
# (152 SMs: 32 lanes up to 608 points, 16 up to 1,216, 8 up to 2,432 and 4 above
# for up to 16 levels; 32 up to 1,216, 16 up to 2,432 and then 8 or 16 above);
# odd counts, the last warp partly empty
@pytest.mark.parametrize("levels,n", [(16, 607), (11, 1215), (16, 2431), (2, 2435), (16, 2435), (17, 1215), (28, 2431),
                                      (28, 2435), (32, 2435), (48, 1219)])
def test_lanes_per_point(mgt, levels, n):
    m = synth.sphere_model(n, levels, 1, 3, seed=50 + levels)
    m.n_coll = m.n_coll * 1e-4
    h = mgt.mgt_model_create(m)
    mgt.mgt_trace_rays(h)
    mgt.mgt_formal_solve(h, want=False)
    got = mgt.mgt_stat_equilibrium(h)
    J, L = mgt.mgt_get_jbar(h)
    p0 = O.lte_populations(m.temp, m.n_spec, m.lines.energy_J, m.lines.g)
    ref = O.stat_equilibrium(p0, J.T, L.T, m.temp, m.n_coll, m.n_spec, m.lines)
    assert np.max(np.abs(got - ref) / np.abs(ref)) < 1e-8


def test_batch_at_the_shared_memory_limit(mgt):
    # 64 levels x 340 lines: three warps of the batched kernel hold 232,320 of the
    # 232,448 bytes of shared memory that a CTA may use, and the kernel's copy of
    # a model's arguments takes 144 more
    levels, n_lines = 64, 340
    m = synth.sphere_model(40, levels, 1, 3, seed=9)
    ln = m.lines
    pairs = np.array([(u, l) for u in range(levels) for l in range(u)], np.int32)[-n_lines:]
    ln.up, ln.lo = np.ascontiguousarray(pairs[:, 0]), np.ascontiguousarray(pairs[:, 1])
    ln.freq_Hz = 1e11 * 1.02 ** np.arange(n_lines)
    ln.A = np.full(n_lines, 1e-6)
    m.n_coll = m.n_coll * 1e-4
    h = mgt.mgt_model_create(m)
    mgt.mgt_trace_rays(h)
    b = mgt.mgt_batch_create([h])
    mgt.mgt_batch_formal_solve(b)
    mgt.mgt_batch_stat_equilibrium(b)
    J, L = mgt.mgt_get_jbar(h)
    p0 = O.lte_populations(m.temp, m.n_spec, ln.energy_J, ln.g)
    ref = O.stat_equilibrium(p0, J.T, L.T, m.temp, m.n_coll, m.n_spec, ln)
    got = mgt.mgt_get_populations(h)
    assert np.max(np.abs(got - ref) / np.abs(ref)) < 1e-8
