"""The per-point kernels (LTE populations, line data, species-density change)
at the edges of their blocks, through the C-ABI against the oracle.

LTE and the rescaled populations are a few FP64 operations: 1e-13 relative.  The
line data are seen through the FP64 formal solution, whose tolerance is the
parity tests' 1e-10.
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


# points around the blocks of 16 (LTE) and 32 (line data); lines around the
# padding to 8, and 17 levels with every pair a line (136: more slots per point
# than half a block of threads), 24 levels (276: more than a block; those rows
# do not fit the staged kernel, the gather kernel takes them)
@pytest.mark.parametrize("n,levels,dense", [(15, 2, False), (31, 9, False), (32, 10, False), (33, 64, False),
                                            (97, 17, False), (40, 17, True), (33, 24, True)])
def test_block_edges(mgt, n, levels, dense):
    m = synth.sphere_model(n, levels, 1, 3, seed=200 + n)
    ln = m.lines
    if dense:
        # one line per level pair, at distinct frequencies far apart
        up, lo = np.array([(u, l) for u in range(levels) for l in range(u)], np.int32).T
        ln.up, ln.lo = np.ascontiguousarray(up), np.ascontiguousarray(lo)
        ln.freq_Hz = 1e11 * 1.02 ** np.arange(len(up))
        ln.A = np.full(len(up), 1e-6)
    h = mgt.mgt_model_create(m)
    if ln.n_lines > 200:
        mgt.mgt_set_solve_opts(h, schedule=1)
    mgt.mgt_trace_rays(h)
    p0 = O.lte_populations(m.temp, m.n_spec, ln.energy_J, ln.g)
    got = mgt.mgt_get_populations(h)
    assert np.max(np.abs(got - p0) / p0) < 1e-13
    J, L = mgt.mgt_formal_solve(h, mgt.MGT_FP64)
    chi, S, _ = O.line_chi_S(p0, ln)
    Jo, Lo = O.formal_solve(m, O.trace(m), chi, S)
    assert np.max(np.abs(J.T - Jo) / Jo) < 1e-10
    assert np.max(np.abs(L.T - Lo) / np.maximum(Lo, 1e-30)) < 1e-10
    Jf, _ = mgt.mgt_formal_solve(h)
    assert np.max(np.abs(Jf.T - Jo) / Jo) < 1e-4
    new = m.n_spec * np.exp(np.random.default_rng(n).normal(size=n))
    mgt.mgt_set_point_fields(h, n_spec=new)
    scaled = mgt.mgt_get_populations(h)
    ref = got * (new / m.n_spec)[:, None]
    assert np.max(np.abs(scaled - ref) / ref) < 1e-13


# lanes per point of the LTE kernel: eight up to 64 points per SM (4,864 on 152
# SMs), above that one for up to 16 levels and two for more; the last block
# full, with one point, partly filled.  The arithmetic does not depend on it:
# every population is that of the same points in a model of half the size, bit
# for bit, down to levels that underflow
@pytest.mark.parametrize("n,levels", [(4864, 16), (4865, 2), (4993, 16), (5000, 17), (4929, 64)])
def test_lte_lanes_per_point(mgt, n, levels):
    rng = np.random.default_rng(n)
    nbrs = np.stack([np.arange(1, n + 1) % n, np.arange(-1, n - 1) % n], axis=1)
    m = synth.Model("ring", rng.uniform(-1, 1, (n, 3)) * 1e11, np.zeros((n, 3)), rng.uniform(5.0, 500.0, n),
                    np.full(n, 1e4), np.full(n, 1e10), rng.uniform(1e3, 1e6, n), 2 * np.arange(n + 1, dtype=np.int64),
                    np.sort(nbrs, axis=1).astype(np.int32).ravel(), np.array([0], np.int32),
                    synth.healpix_directions(1), 3, synth.linear_rotor(levels, rng))
    got = mgt.mgt_get_populations(mgt.mgt_model_create(m))
    for half in (slice(0, n // 2), slice(n // 2, n)):
        k = half.stop - half.start
        nb = np.stack([np.arange(1, k + 1) % k, np.arange(-1, k - 1) % k], axis=1)
        part = synth.Model("part", m.pos[half], m.vel[half], m.temp[half], m.vturb2[half], m.n_coll[half],
                           m.n_spec[half], 2 * np.arange(k + 1, dtype=np.int64),
                           np.sort(nb, axis=1).astype(np.int32).ravel(), np.array([0], np.int32), m.dirs, 3, m.lines)
        np.testing.assert_array_equal(mgt.mgt_get_populations(mgt.mgt_model_create(part)), got[half])
