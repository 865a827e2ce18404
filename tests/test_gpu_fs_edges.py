"""The formal solution at the edges of its chunks, rows per reciprocal and shared
memory, through the C-ABI against the oracle (tolerances of the parity tests:
FP64 1e-10, FP32-mixed 1e-4).
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


def _check(mgt, h, m, precision, tol):
    p0 = O.lte_populations(m.temp, m.n_spec, m.lines.energy_J, m.lines.g)
    chi, S, _ = O.line_chi_S(p0, m.lines)
    J, L = O.formal_solve(m, O.trace(m), chi, S)
    Jg, Lg = mgt.mgt_formal_solve(h, precision)
    assert np.max(np.abs(Jg.T - J) / J) < tol
    assert np.max(np.abs(Lg.T - L) / np.maximum(L, 1e-30)) < tol


# half-rays of every length from 0 to n - 1: remainders of the two and eight
# rows per reciprocal and of the 30-step chunks; thin, thick, and so thick that
# the one-row form takes over.  5 levels: coefficients in registers; 11 levels:
# the shared pre-pass, with an even and an odd number of bins
@pytest.mark.parametrize("levels,bins", [(5, 7), (11, 7), (11, 8), (11, 1)])
@pytest.mark.parametrize("density", [1e-4, 1.0, 1e6])
def test_half_rays_of_every_length(mgt, levels, bins, density):
    n = 75
    rng = np.random.default_rng(levels + bins)
    x = np.linspace(-1, 1, n)
    pos = np.stack([x, 0.05 * x ** 2, 0.02 * np.sin(3 * x)], axis=1)
    nbrs = [[j for j in (i - 1, i + 1) if 0 <= j < n] for i in range(n)]
    off = np.concatenate([[0], np.cumsum([len(v) for v in nbrs])]).astype(np.int64)
    # velocity steps below and above the switch of 0.35 line widths
    vel = np.cumsum(rng.normal(size=(n, 3)) * 600.0, axis=0)
    m = synth.Model("chain", pos * 1e13, vel, 50.0 + 10 * rng.uniform(size=n), np.full(n, 1e6), np.full(n, 1e10),
                    np.full(n, 1e9 * density), off, np.concatenate(nbrs).astype(np.int32),
                    np.array([0, n - 1], np.int32), synth.healpix_directions(1), bins, synth.linear_rotor(levels, rng))
    h = mgt.mgt_model_create(m)
    mgt.mgt_trace_rays(h)
    _check(mgt, h, m, mgt.MGT_FP64, 1e-10)
    _check(mgt, h, m, mgt.MGT_FP32_MIXED, 1e-4)


@pytest.mark.parametrize("n_lines", [328, 330, 336])
def test_lines_at_the_shared_memory_limit(mgt, n_lines):
    # 329 to 336 lines x 11 bins x 48 rays filled a CTA's shared memory to
    # 232,336 of 232,448 bytes with two buffers of step records: with the third
    # they take fewer line groups per CTA
    rng = np.random.default_rng(1)
    levels = 27
    m = synth.sphere_model(30, levels, 2, 11, seed=9)
    ln = m.lines
    pairs = np.array([(u, l) for u in range(levels) for l in range(u)], np.int32)[:n_lines]
    ln.up, ln.lo = np.ascontiguousarray(pairs[:, 0]), np.ascontiguousarray(pairs[:, 1])
    ln.freq_Hz = 1e11 * 1.02 ** np.arange(n_lines)
    ln.A = np.full(n_lines, 1e-6)
    h = mgt.mgt_model_create(m)
    mgt.mgt_set_solve_opts(h, lines_per_thread=8, schedule=2)
    mgt.mgt_trace_rays(h)
    _check(mgt, h, m, mgt.MGT_FP32_MIXED, 1e-4)
