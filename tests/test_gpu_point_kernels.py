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
